"""Rows at the upper end of the fixed-point transforms' range: a single entry just below a power of two, so that the whole
row's scale sits in one value and its twiddled products are as large as they get (listed: entries whose products
overflowed 64 bits when the factors' lower parts went up to 2^31, found by restating the passes in exact integers), and all
positions beside them; in launches small and large enough for either plan.  And the size of the error on random rows.

Tolerances.  One entry v: it is exact, |v| is at least 2^60 units; a pass rounds at most a dozen times by a unit or less (7
passes: 84 units, 2^-53.6 |v|), the output each component by 2^-53 of it: below 2^-52 |v|, taken as 2^-51.  Random rows: 2^-53 at the
output and the roundings of a pass, independent, as one unit of 2^-60 of the row's sum of components each, relative to the
2-norm (at 2187 points two bits fewer in the scale exceed it)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROWS = [
    (81, -1, 66, 1.9842541512957734, 0), (81, -1, 51, 1.964867017371742, 0), (81, 1, 17, 0, 1.9876685343000147),
    (135, 1, 103, 0, 1.9719045237723172), (135, 1, 17, 0, 1.9990958217963104),
    (243, 1, 28, 0, 1.9911539733163754), (243, 1, 95, -1.9971827166857647, 0), (243, -1, 233, 1.9750363750274378, 0),
    (243, 1, 113, 0, 1.9883677494468972), (405, 1, 149, 1.9780459170189026, 0), (405, -1, 67, 1.964867017371742, 0),
    (567, -1, 148, -1.9734099572058563, 0), (567, 1, 95, 1.984879857357891, 0), (567, 1, 42, -1.9852326179224995, 0),
    (625, -1, 379, -1.9940622785931725, 0), (729, -1, 28, 0, -1.9967668796638129), (729, 1, 573, -1.9849531984919391, 0),
    (729, 1, 192, -1.9904181911028247, 0), (2187, -1, 1997, 1.9655409448334249, 0), (2187, 1, 286, 1.9645926751677592, 0),
    (2187, -1, 1048, 1.9654393167763893, 0),
]


def _roots(N, sign):
    ang = np.longdouble("6.283185307179586476925286766559005768") * np.arange(N, dtype=np.longdouble) / N
    return np.cos(ang), sign * np.sin(ang)


@pytest.mark.parametrize("N", sorted({r[0] for r in ROWS}))
@pytest.mark.parametrize("sign", [-1, 1])
def test_one_entry(ctx, N, sign):
    entries = [(p, complex(re, im)) for n, s, p, re, im in ROWS if n == N]
    entries += [(p, v) for p in range(0, N, 1 if N <= 243 else 7) for v in (2 - 2.0 ** -52, -1j * (2 - 2.0 ** -30))]
    x = np.zeros((len(entries), N), dtype=complex)
    for r, (p, v) in enumerate(entries):
        x[r, p] = v
    small = ctx.fft_fibres(torch.as_tensor(x[:8, :, None].copy(), device="cuda"), sign)
    reps = -(-(30000 * 243 // N) // len(entries))
    large = ctx.fft_fibres(torch.as_tensor(x[:, :, None], device="cuda").repeat(reps, 1, 1), sign)
    large = large.reshape(reps, len(entries), N)
    assert torch.equal(large, large[:1].expand_as(large))
    c, s = _roots(N, sign)
    for got in (small[:, :, 0].cpu().numpy(), large[0].cpu().numpy()):
        for r in range(got.shape[0]):
            p, v = entries[r]
            j = np.arange(N) * p % N
            re, im = v.real * c[j] - v.imag * s[j], v.real * s[j] + v.imag * c[j]
            err = np.sqrt((got[r].real - re) ** 2 + (got[r].imag - im) ** 2).max()
            assert err <= 2.0 ** -51 * abs(v), (r, p, v, float(err))


@pytest.mark.parametrize("N", [243, 729, 2187])
@pytest.mark.parametrize("rows", [4, 8000])
def test_random_rows(ctx, N, rows):
    rng = np.random.default_rng(N)
    x = rng.standard_normal((4, N)) + 1j * rng.standard_normal((4, N))
    xt = torch.as_tensor(x[:, :, None], device="cuda").repeat(rows // 4, 1, 1)
    got = ctx.fft_fibres(xt, -1)[:4, :, 0].cpu().numpy()
    c, s = _roots(N, -1)
    j = np.outer(np.arange(N), np.arange(N)) % N
    re, im = x.real @ c[j] - x.imag @ s[j], x.real @ s[j] + x.imag @ c[j]
    passes = round(np.log(N) / np.log(3))
    for r in range(4):
        norm = np.sqrt((re[r] ** 2 + im[r] ** 2).sum())
        err = np.sqrt((got[r].real - re[r]) ** 2 + (got[r].imag - im[r]) ** 2)
        total = (abs(x[r].real) + abs(x[r].imag)).sum()
        bound = 2.0 ** -53 + np.sqrt(passes) * 2.0 ** -60 * total * np.sqrt(N) / norm
        assert np.sqrt((err ** 2).sum()) / norm <= bound, float(np.sqrt((err ** 2).sum()) / norm / bound)
