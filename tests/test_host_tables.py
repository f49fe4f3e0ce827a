"""The tables that the edge kernels read (quadratic pieces of the amplitudes, and of envelope times amplitude) against the
cubic pieces they are derived from, on the host."""

import numpy as np
import pytest
import torch

from oracle import dpa4c as orc
from paper_2608_19041_b200 import binding
from workloads import SMALL_PROFILES, make_blob
from workloads.weights import HEADER_BYTES, blob_array_shapes

U24 = 2.0 ** -24


def _envelope(rho, rc):
    x = rho / rc
    u = 1 - x
    return u ** 4 * (1 + x * (4 + x * (10 + x * (20 + 35 * x)))), -280 * x ** 4 * u ** 3 / rc


def _cubic(m, p, a, b, rho):
    """psi and (chi psi)' of the pair from the cubic pieces and the pair cache."""
    g, dg = m.eval_radial_table(rho)
    pm = m.eval_pair_cache(a, b)
    C0 = p["C0"]
    psi, dpsi = pm[0] * g[:, :C0] + pm[1], pm[0] * dg[:, :C0]
    for q in range(p["R"]):
        psi = psi + pm[2 + q] * g[:, C0 + q:C0 + q + 1]
        dpsi = dpsi + pm[2 + q] * dg[:, C0 + q:C0 + q + 1]
    chi, dchi = _envelope(rho, p["rc"])
    return psi, chi[:, None] * dpsi + dchi[:, None] * psi


def _radii(p, dx):
    rho = np.random.default_rng(0).uniform(0.0, p["rc"], 4000)
    k = np.arange(1, 400) * (dx / 4)                    # joints of whole, halved and quartered intervals
    return np.concatenate([rho, [0.0, 1e-9, p["rc"] - 1e-9], k - 1e-12, k + 1e-12])


def _distance(m, p, per_pair, dx):
    """Largest distances from the cubic pieces, in units of 2^-24 of the largest magnitude."""
    rho, worst = _radii(p, dx), [0.0, 0.0]
    for a in range(p["T"]):
        for b in range(p["T"]):
            got, ref = m.eval_edge_tables(a, b, rho, per_pair), _cubic(m, p, a, b, rho)
            for k in range(2):
                worst[k] = max(worst[k], np.abs(got[k] - ref[k]).max() / (U24 * np.abs(ref[k]).max()))
    return worst


def _steep_blob(p, seed, small, top):
    """A radial map of a large smooth part and a small one of high frequency, and pairs that add nothing to it."""
    blob, at = bytearray(make_blob(p, seed)), HEADER_BYTES
    for name, shape in blob_array_shapes(p):
        n = 4 * int(np.prod(shape))
        w = np.frombuffer(bytes(blob[at:at + n]), dtype="<f4").reshape(shape).copy()
        if name == "X0":
            w[:] = 0.0
        if name == "omega":
            w[-1] = top
        if name == "W_in":
            w[1:-1] = 0.0
            w[-1] *= small
        blob[at:at + n] = w.astype("<f4").tobytes()
        at += n
    return bytes(blob)


# Pieces are cut until psi is within 1 and the product within 2 units of 2^-24 of their largest magnitude; the leading
# coefficient's rounding adds half a unit, and where gamma g, beta and U q cancel, the sum of the parts' errors
# meets a smaller magnitude.  Against the shared tables, which come from the map itself, the cubic pieces' own packed words
# add up to a unit of value and two of derivative at the default spacing (their share grows with the spacing).
PSI, PRODUCT = 3.0, 5.0


@pytest.mark.parametrize("basis", ["bessel", "gaussian"])
@pytest.mark.parametrize("name,dx,per_pair", [
    ("p8_2_0", 0.002, 0), ("p8_2_0", 0.002, 1), ("p16_3_2", 0.002, 0), ("p16_3_2", 0.002, 1), ("p32_2_0_res", 0.002, 0),
    ("p32_2_0_res", 0.002, 1), ("p32_2_4", 0.002, 0), ("p32_2_4", 0.002, 1), ("p32_2_4", 0.05, 1), ("p64_3_8", 0.002, 1),
    ("p128_2_0", 0.002, 0), ("p128_2_0", 0.002, 1), ("p128_2_0", 0.01, 1)])
def test_edge_tables_follow_the_cubic_pieces(name, dx, per_pair, basis):
    p = SMALL_PROFILES[name]
    m = binding.Model(make_blob(p, seed=5, basis=basis), table_dx=dx)
    psi, product = _distance(m, p, per_pair, dx)
    assert psi <= PSI and product <= PRODUCT


def test_a_steep_map_with_shared_modes_is_cut_for_the_products_too():
    # a large smooth part and a small one of high frequency: the values are within their bound long before the products
    p = SMALL_PROFILES["p32_2_4"]
    m = binding.Model(_steep_blob(p, 3, 3e-6, 250))
    psi, product = _distance(m, p, 1, 0.002)
    assert psi <= PSI and product <= PRODUCT


@pytest.mark.parametrize("basis", ["bessel", "gaussian"])
@pytest.mark.parametrize("name", ["p64_3_8", "p128_2_0", "p128_3_4"])
def test_splines_follow_the_radial_map_between_the_knots(name, basis):
    p = SMALL_PROFILES[name]
    blob = make_blob(p, seed=5, basis=basis)
    m, o = binding.Model(blob), orc.Oracle(blob)        # (fitted when the model is made: no list build waits for it)
    rho = torch.from_numpy(np.random.default_rng(1).uniform(1e-3, p["rc"], 3000)).requires_grad_(True)
    g, q = orc.radial_map(rho, o.prm, o.p.get("basis", "bessel"), o.p["rc"])
    gs = [torch.autograd.grad(c.sum(), rho, retain_graph=True)[0].numpy() for c in torch.cat([g, q], dim=1).T]
    y, dy = torch.cat([g, q], dim=1).detach().numpy(), np.stack(gs, axis=1)
    C0 = p["C0"]
    for t in range(p["T"]):
        gamma, beta, U = (x[t, t].numpy() for x in o.pair)
        psi, dpsi = gamma * y[:, :C0] + beta, gamma * dy[:, :C0]
        if p["R"]:
            psi, dpsi = psi + y[:, C0:] @ U.T, dpsi + dy[:, C0:] @ U.T
        got = m.eval_edge_splines(t, rho.detach().numpy())
        # the fit's bounds, 2^-24 and 2^-23 of the largest, one more for gamma, beta and U in single precision, and the coefficients'
        # own 2^-25: of the value half a unit, of the slope 32 of their differences per Angstrom against a slope of about twice the value
        assert np.abs(got[0] - psi).max() <= 3 * U24 * np.abs(psi).max()
        assert np.abs(got[1] - dpsi).max() <= 3 * 2 * U24 * np.abs(dpsi).max() + 32 * U24 * np.abs(psi).max()


def test_narrow_models_have_no_splines():
    m = binding.Model(make_blob(SMALL_PROFILES["p32_2_4"], seed=5))
    with pytest.raises(binding.UmlmdError, match="splines"):
        m.eval_edge_splines(0, [1.0])


def test_splines_at_the_ends_and_at_no_number():
    p = SMALL_PROFILES["p128_2_0"]
    m = binding.Model(make_blob(p, seed=5))
    psi, dpsi = m.eval_edge_splines(1, [-1.0, 0.0, p["rc"], 2 * p["rc"], np.nan, -np.nan])
    assert np.array_equal(psi[0], psi[1]) and np.array_equal(psi[2], psi[3]) and np.isfinite(psi[:4]).all() and np.isfinite(dpsi[:4]).all()
    assert np.isnan(psi[4:]).all() and np.isnan(dpsi[4:]).all()


@pytest.mark.parametrize("name", ["p64_3_8", "p128_2_0"])
def test_splines_have_no_common_factor(name):
    p = SMALL_PROFILES[name]
    blob = make_blob(p, seed=84)
    m, o = binding.Model(blob), orc.Oracle(blob)
    rho = np.random.default_rng(2).uniform(1.0, p["rc"], 3000)
    with torch.no_grad():
        g, q = (x.numpy() for x in orc.radial_map(torch.from_numpy(rho), o.prm, o.p.get("basis", "bessel"), o.p["rc"]))
    gamma, beta, U = (x[0, 0].numpy() for x in o.pair)
    psi = gamma * g + beta + (q @ U.T if p["R"] else 0.0)
    got = m.eval_edge_splines(0, rho)[0]
    # gamma, beta and U of the pair are rounded by up to 2^-25, at random over the dozen channels and more that carry them
    assert abs((got * psi).sum() / (psi * psi).sum() - 1) <= 8e-9
