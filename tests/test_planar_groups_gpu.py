"""Planar windows where a CTA of the row-FFT kernel holds several subbands: all
of them in one turn of its entry table, two turns, one vector and two per
subband, training and test vectors side by side, a last CTA that is not full;
and the calls that go to the general kernel instead (three turns, few
vectors).  Reference and tolerances are test_planar_fft_gpu's."""
import pytest

import paper_2508_11790_gb300 as P
import test_planar_fft_gpu as planar

pytestmark = pytest.mark.gpu

FOUR = [(4, 2), (2, 4), (1, 1), (3, 3)]


@pytest.mark.parametrize("Nx,Nz,Mx,Mz,F,L,win,K,prec,shard", [
    (5, 3, 8, 16, 256, 256, [(3, 5), (2, 2)], [2, 1], P.BS_PREC_FP32, None),          # 32 subbands, one turn
    (32, 4, 32, 4, 512, 256, FOUR * 5, [3, 2, 4, 1] * 5, P.BS_PREC_FP16, None),       # 16 subbands, two turns
    (16, 8, 16, 8, 512, 256, FOUR * 10, [3] * 40, P.BS_PREC_FP32, None),              # three turns: general
    (32, 4, 64, 8, 64, 64, FOUR, [1, 2, 1, 2], P.BS_PREC_BF16, None),                 # 8 subbands of one vector
    (32, 2, 32, 4, 1024, 512, FOUR, [3, 1, 2, 4], P.BS_PREC_FP32, (8, 8)),            # a shard: few vectors
    (30, 2, 64, 4, 256, 256, FOUR, [2, 1, 1, 2], P.BS_PREC_FP32, (64, 8)),            # 8 vectors a record of 16 a CTA
    (8, 8, 8, 16, 64, 4, FOUR, [20, 5, 16, 33], P.BS_PREC_FP32, None),                # 256 vectors: general
    (8, 8, 8, 16, 128, 8, FOUR, [30, 5, 16, 33], P.BS_PREC_FP16, None)])              # 640: two subbands a CTA
def test_planar_windows_of_several_subbands(Nx, Nz, Mx, Mz, F, L, win, K, prec, shard):
    planar.test_planar_windows(Nx, Nz, Mx, Mz, F, L, win, K, prec, shard)
