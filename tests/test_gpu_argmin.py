"""poseidon_argmin and poseidon_argmin_noalloc at the sizes and alignments
where their kernels change path: 16-entry words and their remainder, the
one-block limit (16384 entries), buffers off the 16-byte alignment."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift_T,shift_F", [(0, 0), (1, 0), (0, 1), (4, 16), (3, 7)])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 255, 4095, 4096, 4097, 16383, 16384, 16385,
                               16401, 70_001, 2_500_007])
def test_argmin_paths(n, shift_T, shift_F):
    import torch

    import paper_2609_06086_gb300 as P
    rng = np.random.default_rng(n)
    big = np.iinfo(np.int32).max
    for share in (0.0, 2.0 / n, 0.5, 1.0):
        # codes 0..3 and neighbours of 1 in every bit; ties and extremes
        F = rng.choice(np.array([0, 2, 3, 128, 129, 255], np.uint8), n)
        F[rng.random(n) < share] = 1
        T = rng.choice(np.array([0, 1, big - 1, big, -1], np.int32), n)
        T[F == 1] = rng.choice(np.array([7, 8, big - 1, big], np.int32), int((F == 1).sum()))
        dT = torch.zeros(n + shift_T, dtype=torch.int32, device="cuda")
        dF = torch.ones(n + shift_F, dtype=torch.uint8, device="cuda")
        dT[shift_T:] = torch.from_numpy(T).cuda()
        dF[shift_F:] = torch.from_numpy(F).cuda()
        idx = np.flatnonzero(F == 1)
        want = -1 if len(idx) == 0 else int(idx[np.argmin(T[idx])])
        out = torch.full((2,), -9, dtype=torch.int64, device="cuda")
        s = torch.cuda.current_stream().cuda_stream
        a, b = dT[shift_T:].data_ptr(), dF[shift_F:].data_ptr()
        P.poseidon_argmin(a, b, n, out.data_ptr(), s)
        P.binding.poseidon_argmin_noalloc(a, b, n, out[1:].data_ptr(), s)
        torch.cuda.synchronize()
        assert out.tolist() == [want, want], (n, share)
