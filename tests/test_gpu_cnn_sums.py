"""The proposal network's training kernel with many samples per CTA: the error of the
gradients' summation, and calls of every shape against the FP64 network."""
import ctypes
import math

import numpy as np
import pytest

import synthetic
from oracle import cnn
from tests.test_gpu_parity import mr  # noqa: F401

pytestmark = pytest.mark.gpu

W_POS = 4.0


def samples(Bs, n, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    T = Bs + 8
    x = torch.empty(n, 2, T, T)
    x[:, 0] = torch.rand(n, T, T, generator=g) * 2 - 1
    x[:, 1] = torch.rand(n, T, T, generator=g) * 3 - 3
    return x, (torch.rand(n, generator=g) < 0.1).float()


def weights(seed):
    rng = np.random.default_rng(seed)
    return synthetic.cnn_init_params(cnn.SHAPES, seed=seed) + 0.02 * rng.standard_normal(cnn.NPARAM)


@pytest.mark.parametrize("Bs,ctas", [(17, 2), (33, 1)])
def test_summation_error_over_the_samples_of_a_cta(mr, Bs, ctas):  # noqa: F811
    # 2048 samples on the CTAs of one SM, against the FP64 sum of the kernel's own
    # gradients of one sample per CTA.  The mean's factor 1/n is a power of two, so both
    # add the same numbers and only the sum over a CTA's k = n / ctas samples differs.
    # An addition rounds a running sum S_i by u |S_i| / sqrt(3) or less (rms,
    # u = 2^-24); S_i / S grows like sqrt(i / k) for terms of random sign (less slowly for
    # terms of one sign), so the k roundings add up to u sqrt(k / 2) / sqrt(3) of the
    # gradient, and those of independent CTAs to 1 / sqrt(ctas) of that.  Norms over
    # the 288 or 2304 weights of a layer stay within 1.5 times that.
    import torch
    n, k = 2048, 2048 // ctas
    tol = 1.5 * 2.0 ** -24 * math.sqrt(k / 2) / math.sqrt(3) / math.sqrt(ctas)
    train = getattr(mr.load_library(), "_ZN2mr12launch_trainEiPKfS1_PKiliS1_fPfS4_S4_iP11CUstream_st")
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    x, y = (t.cuda() for t in samples(Bs, n, 100))
    w = torch.from_numpy(weights(9).astype(np.float32)).cuda()

    def grad(s0, nb, out):  # samples s0 .. s0 + nb - 1, CTAs of one SM
        train(ctypes.c_int(Bs), ptr(x), ptr(y), None, ctypes.c_int64(s0), ctypes.c_int(nb), ptr(w),
              ctypes.c_float(W_POS), ptr(out), None, None, ctypes.c_int(1), None)

    got = torch.zeros(cnn.NPARAM, device="cuda")
    grad(0, n, got)
    want = torch.zeros(cnn.NPARAM, dtype=torch.float64, device="cuda")
    part = torch.zeros(cnn.NPARAM, device="cuda")
    for s0 in range(0, n, ctas):
        part.zero_()
        grad(s0, ctas, part)
        want += part.double() / k
    torch.cuda.synchronize()
    got, want = got.double().cpu().numpy(), want.cpu().numpy()
    for a, b in zip(cnn.unpack(got), cnn.unpack(want)):
        if a.ndim == 4:
            assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), (a.shape, np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [1, 7, "several"])
@pytest.mark.parametrize("Bs", [17, 33])
def test_calls_of_every_shape_match_fp64_reference(mr, Bs, n):  # noqa: F811
    # one sample (a CTA of a cluster has none), fewer than CTAs, and three or more for
    # every CTA with an odd rest; five tiled samples, so that the reference is their
    # weighted mean.  Bounds as for six samples of 25^2: FP32 arithmetic against FP64,
    # probabilities to 1e-5, loss and gradient to 1e-4 of the gradient's scale
    import torch
    if n == "several":
        n = 2 * 3 * torch.cuda.get_device_properties(0).multi_processor_count + 3
    g = mr.Forest(dim=2, Bs=Bs, trees=[dict(Jmin=2, Jmax=4, ic="none")], capacity=1000)
    theta, rng, T = weights(9), np.random.default_rng(4), Bs + 8
    m = min(n, 5)
    base, label = rng.standard_normal((m, 2, T, T)), np.array([1, 0, 1, 1, 0], np.float64)[:m]
    of = np.arange(n) % m
    share = np.bincount(of) / n
    p, gr, loss = g.cnn_eval(theta, base[of], label[of], w_pos=W_POS)
    pref = np.array([cnn.forward(theta, x)[0] for x in base])
    ref = [cnn.loss_and_grad(theta, [x], [y], W_POS) for x, y in zip(base, label)]
    L, gref = sum(a * r[0] for a, r in zip(share, ref)), sum(a * r[1] for a, r in zip(share, ref))
    np.testing.assert_allclose(p, pref[of], rtol=0, atol=1e-5)
    assert abs(loss - L) <= 1e-4 * max(1.0, abs(L))
    assert np.abs(gr - gref).max() <= 1e-4 * np.abs(gref).max(), np.abs(gr - gref).max()
