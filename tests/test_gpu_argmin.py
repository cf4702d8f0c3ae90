"""poseidon_argmin and poseidon_argmin_noalloc at the sizes and alignments
where their kernels change path: 16-entry words and their remainder, the
one-block limits (16384 entries, 1024 off the 16-byte alignment), buffers off
that alignment."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift_T,shift_F", [(0, 0), (1, 0), (0, 1), (4, 16), (3, 7)])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 255, 1024, 1025, 4095, 4096, 4097, 16383, 16384, 16385,
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


def test_unaligned_buffers_are_not_left_to_one_block():
    """16384 entries that have to be read one by one take less time than
    aligned ones (two and a half times as long when one block reads them)."""
    import torch

    import paper_2609_06086_gb300 as P
    n = 16384
    T = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    F = torch.ones(n + 1, dtype=torch.uint8, device="cuda")
    out = torch.zeros(1, dtype=torch.int64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream

    def time_of(shift):
        best = float("inf")
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(200):
                P.binding.poseidon_argmin_noalloc(T[shift:].data_ptr(), F[shift:].data_ptr(), n,
                                                  out.data_ptr(), s)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert time_of(1) < 1.8 * time_of(0)
