"""Products of several vectors whose images do not fit shared memory together and go
in passes of half as many with one correlator kernel: reference and tolerance of
test_gpu_pass.py."""
import pytest

import test_gpu_pass as whole

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lx,ly,nu,nd,corr,n", [
    (7, 6, 10, 10, "2x2", 700), (10, 6, 8, 6, "pair", 257), (10, 6, 15, 15, "2x2", 33), (8, 8, 9, 7, "none", 300)])
def test_groups_of_vectors(lx, ly, nu, nd, corr, n):
    whole.test_products_and_means_of_the_stored_values(lx, ly, nu, nd, corr, n)
