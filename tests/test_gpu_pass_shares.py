"""The passes with FP64 sums where the number of images and of their owners changes: few
elements per sample, the sizes at which an owner's share doubles, and sample sets
too small for more images.  Reference and tolerance of test_gpu_pass.py."""
import pytest

import test_gpu_pass as whole

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lx,ly,nu,nd,corr,n", [
    (4, 4, 1, 1, "pair", 3000), (4, 4, 2, 2, "2x2", 9), (5, 5, 6, 6, "pair", 4100), (6, 6, 8, 8, "none", 2000),
    (6, 6, 9, 7, "pair", 700), (6, 6, 9, 9, "2x2", 1500), (6, 6, 12, 12, "pair", 400),
    (6, 6, 16, 16, "pair", 640), (6, 6, 17, 17, "none", 5000), (8, 5, 18, 18, "pair", 200), (7, 6, 21, 21, "2x2", 90),
    (8, 8, 23, 23, "pair", 600)])
def test_shares_of_the_images(lx, ly, nu, nd, corr, n):
    whole.test_products_and_means_of_the_stored_values(lx, ly, nu, nd, corr, n)
