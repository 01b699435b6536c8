"""The FP64 path's reciprocal of the density, seen through the fields of a uniform
lattice: u_x = f_l j_x (1 / rho), with f chosen so that rho and j_x are exact."""
import numpy as np
import pytest

from paper_1909_13086_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

# f_i = F_i 2^e: rho = R 2^e and j_x = 2^e, exact sums of small integers
WEIGHTS = {3: (1, 1, 0, 0, 1), 4: (1, 2, 0, 1, 0), 5: (2, 1, 1, 0, 1), 7: (3, 2, 1, 1, 0)}  # rho in (2^1, 2^3)


@pytest.fixture(scope="module")
def lattice():
    import torch

    torch.cuda.set_device(0)
    s = torch.cuda.Stream()
    lat = lbm.Lattice(5, 5, workloads.params(Ra=1e4, strip_width=0.0), precision="fp64", stream=s.cuda_stream)
    yield lat
    lat.close()


def velocity(lat, F, e, sign=1.0):
    """(rho, u_x) of the middle cell with f_i = sign F_i 2^e and all cells liquid."""
    f = np.zeros((9, 5, 5))
    for i, v in enumerate(F):
        f[i] = np.ldexp(sign * v, e)
    g = np.full((9, 5, 5), 1.0)  # H = 9 > L
    lat.set_populations(f, g, 0)
    lat.step(1)
    F_ = lat.fields()
    assert F_["fl"][2, 2] == 1.0
    return F_["rho"][2, 2], F_["ux"][2, 2]


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("R", sorted(WEIGHTS))
def test_velocity_over_the_exponent_range(lattice, R, sign):
    """Where the reciprocal takes Newton steps it is within half a unit in the last
    place of 1 / rho and a term of 2^-80, as the quotient is within half a unit: with a
    rounding of the product on either side the velocities differ by less than 4 x 2^-53
    relatively.  From 2^1021 on, where the reciprocal nears the subnormals, and below
    2^-1021 the quotient itself is taken: the same bits."""
    F = WEIGHTS[R]
    jx = float(F[1] - F[3])
    top = int(np.floor(np.log2(R)))
    exps = sorted({*range(-1070, 1020, 37), *range(-1028, -1015), *range(1010, 1024 - top), -1, 0, 1})
    with np.errstate(all="ignore"):
        for e in exps:
            rho, ux = velocity(lattice, F, e, sign)
            assert rho == np.ldexp(sign * R, e), e
            want = np.ldexp(sign * jx, e) * (1.0 / rho)
            at = e + top  # rho in [2^at, 2^(at + 1))
            if at < -1021 or at >= 1021:
                assert ux == want, (e, ux, want)
            else:
                assert abs(ux - want) <= 1.01 * 4 * 2.0 ** -53 * abs(want), (e, ux, want)


@pytest.mark.parametrize("rho", [0.0, -0.0, np.inf, -np.inf, np.nan])
def test_velocity_of_a_density_without_reciprocal(lattice, rho):
    got, ux = velocity(lattice, (rho, 0, 0, 0, 0), 0)
    with np.errstate(all="ignore"):
        want = np.float64(0.0) * (np.float64(1.0) / np.float64(rho))
    assert np.array_equal(got, rho, equal_nan=True) and np.array_equal(ux, want, equal_nan=True)
