"""The dense z operators (tensor-core form of the z derivatives): tables and
geometry on the CPU, the kernel against the oracle and the transform kernel on
the GPU."""
import ctypes

import numpy as np
import pytest

from oracle import fc


def _lib():
    from paper_2002_01392_gb300 import build
    build.build()
    return ctypes.CDLL(build.HOSTCHECK)


@pytest.mark.parametrize("Nz,C", [(10, 25), (33, 25), (32, 25), (39, 25), (103, 25), (104, 25), (129, 25), (231, 33),
                                  (487, 25), (488, 25), (512, 25), (513, 25), (513, 33), (549, 25), (550, 25)])
def test_dense_tables_are_the_derivative_operators(Nz, C):
    """Orbits cover every row once per member; the blocks, put together by the
    kernel's own rules (parts of a line, high + low values per slab, members of
    an output orbit), are the circular derivative operators of the continued grid."""
    lib, Np = _lib(), Nz + C
    o = (ctypes.c_int * 6)()
    assert lib.fchc_dense_geom(Nz, Np, o) == 0
    NQ, No, KQ, NC, chunks, slabs = list(o)
    assert NQ * KQ <= 576 and NC % 16 == 0 and NQ * NC <= 192 and chunks * NC >= No
    rows = np.array([[lib.fchc_dense_row(Nz, Np, j, i) for i in range(NQ)] for j in range(No)])
    assert sorted(set(rows.ravel())) == list(range(Np))
    assert len({tuple(sorted(set(r))) for r in rows}) == No
    x = np.random.default_rng(Nz).standard_normal((Np, 4))
    # members (mirror, shift) and parts (m, s): sign (-1)^(bits of part & member)
    sign = np.array([[(-1.0) ** bin(q & i).count("1") for i in range(NQ)] for q in range(NQ)])
    parts = [sum(sign[q, i] * x[rows[:, i]] for i in range(NQ)) for q in range(NQ)]
    cuts = np.cumsum([0] + [lib.fchc_dense_slab(Nz, Np, s) for s in range(slabs)])
    assert cuts[-1] * 16 == KQ and (np.diff(cuts) > 0).all()
    k = fc.kz_wavenumbers(Nz, C, Nz - 1.0)          # unit spacing
    for order in (1, 2):
        halves = np.zeros(2 * KQ * NC * chunks * NQ, dtype=np.uint16)
        e = ctypes.c_int()
        assert lib.fchc_dense_blocks(Nz, Np, order, halves.ctypes.data_as(ctypes.c_void_p), ctypes.byref(e)) == 0
        v = halves.view(np.float16).astype(np.float64)
        assert np.isfinite(v).all() and 2.0 ** 12 <= np.abs(v).max() <= 2.0 ** 13
        Y = np.zeros((NQ, chunks * NC, 4))
        p = 0
        for ch in range(chunks):
            for q in range(NQ):
                for a, b in zip(cuts, cuts[1:]):
                    n = (b - a) * 16 * NC
                    B = (v[p:p + n] + v[p + n:p + 2 * n]).reshape(2 * (b - a), NC, 8).transpose(1, 0, 2).reshape(NC, -1)
                    p += 2 * n
                    src = np.zeros((KQ, 4))
                    src[:No] = parts[q]
                    Y[q, ch * NC:(ch + 1) * NC] += B @ src[16 * a:16 * b]
        assert p == v.size and not Y[:, No:].any()
        par = -1.0 if order == 1 else 1.0
        y = np.full((Np, 4), np.nan)
        for i in range(NQ):
            y[rows[:, i]] = (par if i & 1 else 1.0) * sum(sign[q, i] * Y[q, :No] for q in range(NQ))
        ref = np.fft.ifft(np.fft.fft(x, axis=0) * fc.deriv_factor(k, order)[:, None], axis=0).real
        # the blocks carry 22 bits and a sign: each entry within 2^-23 of itself or 2^-25 of 1 (scaled to 2^12..2^13)
        y *= 2.0 ** -e.value
        assert np.abs(y - ref).max() < 2.0 ** -22 * np.pi ** order * np.abs(x).max() * np.sqrt(Np)


def test_dense_plans_have_room_for_two_slabs():
    """Every d, C and Nz that fc_setup accepts: the continuation's shared memory leaves two slabs, or the plan has no
    dense operators (and its calls take the transforms)."""
    lib = _lib()
    smem, left_out = ctypes.c_int(), 0
    o = (ctypes.c_int * 6)()
    for d in range(2, 11):
        for C in range(d, 65):
            for Nz in range(2 * d, 577 - C):
                n = lib.fchc_dense_plan(Nz, d, C, ctypes.byref(smem))
                if n:
                    assert 2 <= n <= 8 and smem.value <= 227 * 1024
                else:
                    left_out += lib.fchc_dense_geom(Nz, Nz + C, o) == 0
    assert left_out > 0


# ---------------------------------------------------------------------------
# the kernel (GPU)
# ---------------------------------------------------------------------------
@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2002_01392_gb300 import api as a
    assert torch.cuda.is_available()
    return a


def _oracle(f, Mr, order, Lz=1.0):
    """Derivative of f [Nz][lines] as the dense operator, in float64."""
    return fc.dense_deriv_operator(f.shape[0], Mr.shape[0], Lz, Mr, order) @ f.astype(np.float64)


def _bound(f, Mr, order, Lz=1.0):
    """Rounding of the split operands and of the float32 sums, per line: the operator's entries and the line carry
    2^-23 of their largest magnitudes each, products and sums of a block of at most 36 16-steps 2^-24 per addition,
    all amplified by at most k_max^order over the continued line's 2-norm."""
    xe = fc.extend(f.astype(np.float64), Mr)
    kmax = np.pi * (f.shape[0] - 1) / Lz
    return 16 * 2.0 ** -23 * kmax ** order * np.linalg.norm(xe, axis=0)


# every branch: parts 4 (N' even) and 2 (odd), one and several chunks and slabs, resident blocks, direct lengths, a last
# tile of few lines, a tile across two fields, odd line counts, one output, Lz
@pytest.mark.gpu
@pytest.mark.parametrize("Nz,Ny,Nx,B,Lz", [(104, 363, 121, 3, 1.0), (155, 128, 128, 1, 2.0), (257, 129, 128, 1, 1.0),
                                            (350, 64, 257, 1, 0.5), (487, 317, 311, 1, 1.0), (512, 131, 127, 1, 1.0),
                                            (513, 64, 129, 2, 1.0), (549, 128, 129, 1, 1.0)])
def test_dense_kernel_matches_oracle(api, Mr_5_25, Nz, Ny, Nx, B, Lz):
    import torch
    g = torch.Generator(device="cuda").manual_seed(Nz)
    z = torch.arange(Nz, device="cuda") / (Nz - 1)
    amp = torch.rand((3, B, 1, Ny, Nx), generator=g, device="cuda") * 2 - 1
    zz = z[None, :, None, None]
    f = amp[0] * torch.sin(9 * zz) + amp[1] * torch.cos(31 * zz * amp[2]) * 10
    f[:, ::7] += 1e-3 * torch.rand((B, (Nz + 6) // 7, Ny, Nx), generator=g, device="cuda")
    f = f.contiguous()
    plan = api.Plan(5, 25, Nz)
    d1, d2 = torch.full_like(f, float("nan")), torch.full_like(f, float("nan"))
    api.fc_deriv_z(plan, f, d1, d2, Lz=Lz)
    only = torch.full_like(f, float("nan"))
    api.fc_deriv_z(plan, f, None, only, Lz=Lz)
    torch.cuda.synchronize()
    assert torch.equal(only, d2) and torch.isfinite(d1).all() and torch.isfinite(d2).all()
    lines = lambda t: t.permute(0, 2, 3, 1).reshape(-1, Nz)  # noqa: E731
    n = Ny * Nx * B
    pick = np.unique(np.r_[0:130, n // 2 - 65:n // 2 + 65, n - 140:n])
    fp, o1, o2 = (lines(t)[pick].cpu().numpy().T for t in (f, d1, d2))
    for order, out in ((1, o1), (2, o2)):
        err = np.linalg.norm(out - _oracle(fp, Mr_5_25, order, Lz), axis=0)
        assert (err <= _bound(fp, Mr_5_25, order, Lz)).all(), (order, (err / _bound(fp, Mr_5_25, order, Lz)).max())


@pytest.mark.gpu
def test_dense_kernel_magnitudes_and_nonfinite(api, Mr_5_25):
    """Lines whose sample gives the wrong scale (a peak between sampled rows, zero but for one row), of magnitudes from
    1e-37 to 1e33, of zeros: each to its own bound; a NaN or Inf spoils its own line only.  Entry points that route the
    same call agree bitwise."""
    import ctypes
    import torch
    Nz, Ny, Nx = 513, 8, 2050
    r = np.random.default_rng(5)
    z = np.arange(Nz) / (Nz - 1)
    base = (np.sin(np.outer(z, r.uniform(3, 40, Ny * Nx)) + 1)).astype(np.float32)
    f = base.copy()
    f[:, 0:9] = 0
    f[Nz // 2 + 1, 0:9] = 1e5
    f[:, 9:18] *= 1e-3
    f[Nz // 3 + 1, 9:18] = 1e4
    for i, s in enumerate((1e33, 1e-30, 1e-37)):
        f[:, 18 + 9 * i:27 + 9 * i] *= np.float32(s)
    f[:, 45:54] = 0
    f[5, 300], f[7, 500] = np.nan, np.inf
    ft = torch.from_numpy(f).cuda().view(Nz, Ny, Nx)
    plan = api.Plan(5, 25, Nz)
    d = [torch.empty_like(ft) for _ in range(2)]
    api.fc_deriv_z(plan, ft, *d)
    out = [t.view(Nz, -1).cpu().numpy() for t in d]
    good = np.ones(Ny * Nx, bool)
    good[[300, 500]] = False
    for o in out:
        assert np.isfinite(o[:, good]).all() and not np.isfinite(o[:, ~good]).any()
        assert not o[:, 45:54].any()
    pick = np.r_[0:45, 54:200, 640:700]
    for order in (1, 2):
        err = np.linalg.norm(out[order - 1][:, pick] - _oracle(f[:, pick], Mr_5_25, order), axis=0)
        assert (err <= _bound(f[:, pick], Mr_5_25, order)).all()
    # host arrays in slabs, and the variant without allocations
    h = [torch.empty((Nz, Ny, Nx)) for _ in range(2)]
    api.fc_deriv_z_host(plan, ft.cpu(), *h, slab_bytes=2 * Nz * Nx * 4)
    n = [torch.empty_like(ft) for _ in range(2)]
    assert api._lib.fc_deriv_z_noalloc(plan.handle, api.FC_F32, 1, Nx, Ny, ctypes.c_double(1.0), ft.data_ptr(),
                                       n[0].data_ptr(), n[1].data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    for a, b, c in zip(d, h, n):
        av = a.cpu().view(torch.int32)
        fin = torch.isfinite(a.cpu())
        assert torch.equal(av[fin], b.view(torch.int32)[fin]) and torch.equal(av[fin], c.cpu().view(torch.int32)[fin])


@pytest.mark.gpu
@pytest.mark.parametrize("d,C,Nz", [(5, 60, 500), (10, 64, 480), (7, 64, 461),      # no room for two slabs: transforms
                                    (7, 33, 513), (4, 40, 257), (10, 25, 350), (9, 64, 200)])   # other d and C, N' even and odd
def test_dense_continuations(api, d, C, Nz):
    """Calls of the dense operators' size with other continuations than (5, 25)."""
    import torch
    Ny, Nx = 8, 2049
    r = np.random.default_rng(Nz)
    z = np.arange(Nz) / (Nz - 1)
    f = (np.sin(np.outer(z, r.uniform(3, 40, Ny * Nx)) + 1) + 0.1 * z[:, None] ** 2).astype(np.float32)
    plan = api.Plan(d, C, Nz)
    Mr = plan.matrix()
    ft = torch.from_numpy(f).cuda().view(1, Nz, Ny, Nx)
    out = [torch.empty_like(ft) for _ in range(2)]
    api.fc_deriv_z(plan, ft, *out)
    pick = np.r_[0:128, 8000:8128, Ny * Nx - 129:Ny * Nx]
    for order in (1, 2):
        err = np.linalg.norm(out[order - 1].view(Nz, -1)[:, pick].cpu().numpy() - _oracle(f[:, pick], Mr, order), axis=0)
        assert (err <= _bound(f[:, pick], Mr, order)).all()


def _field_with_peaks(Nz, n, seed):
    """Smooth lines of magnitude about 1; every 37th has a peak of 300 to 3e5 on a row between two sampled ones."""
    r = np.random.default_rng(seed)
    z = np.arange(Nz) / (Nz - 1)
    f = np.sin(np.outer(z, r.uniform(3, 40, n)) + 1)
    at = np.arange(0, n, 37)
    every = (Nz + 31) // 32
    f[r.integers(1, Nz // every - 1, at.size) * every + r.integers(1, every, at.size), at] = 10.0 ** r.uniform(2.5, 5.5, at.size)
    return f.astype(np.float32)


@pytest.mark.gpu
@pytest.mark.parametrize("Nz", [513, 350])
def test_dense_kernel_reloaded_tiles(api, Mr_5_25, Nz):
    """Tiles whose sampled scale turns out too small are loaded twice: every line to its own bound, the same bits in
    repeated calls."""
    import torch
    Ny, Nx = 8, 2560
    f = _field_with_peaks(Nz, Ny * Nx, Nz)
    ft = torch.from_numpy(f).cuda().view(1, Nz, Ny, Nx)
    plan = api.Plan(5, 25, Nz)
    d = [torch.empty_like(ft) for _ in range(2)]
    e = [torch.empty_like(ft) for _ in range(2)]
    api.fc_deriv_z(plan, ft, *d)
    for _ in range(5):
        api.fc_deriv_z(plan, ft, *e)
        assert torch.equal(d[0], e[0]) and torch.equal(d[1], e[1])
    for order in (1, 2):
        err = np.linalg.norm(d[order - 1].view(Nz, -1).cpu().numpy() - _oracle(f, Mr_5_25, order), axis=0)
        assert (err <= _bound(f, Mr_5_25, order)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("Nz,lines", [(129, 131072), (512, 16384), (513, 16384), (520, 16384)])
def test_dense_kernel_is_no_less_exact_than_the_transforms(api, Nz, lines):
    """Rough lines (an inertial-range spectrum, smooth at the walls): the error against the float64 derivatives, in the
    2-norm, of the dense operators and of the transforms, which a call of few lines takes."""
    import torch
    r = np.random.default_rng(Nz)
    z = np.arange(Nz) / (Nz - 1)
    k = np.arange(1, 2 * (Nz - 1) // 3 + 1)
    i = np.minimum(np.arange(Nz), np.arange(Nz)[::-1])
    damp = np.sin(0.5 * np.pi * np.clip((i - 5) / 10, 0, 1)) ** 2
    prof = [damp * (k[:, None] ** (-5 / 6) * np.cos(np.pi * np.outer(k, z) + 2 * np.pi * r.random((k.size, 1)))).sum(0)
            + np.cos(r.uniform(1, 9) * z + r.uniform(0, 6)) for _ in range(8)]
    f = torch.from_numpy((np.array(prof).T @ r.standard_normal((8, lines))).astype(np.float32)).cuda().view(1, Nz, 1, lines)
    part = f[..., :4096].contiguous()
    plan = api.Plan(5, 25, Nz)
    outs = []
    for x in (f, part, part.double()):
        o = [torch.empty_like(x) for _ in range(2)]
        api.fc_deriv_z(plan, x, *o)
        outs.append([t[..., :4096].double() for t in o])
    for dense, transform, exact in zip(*outs):
        assert not torch.equal(dense, transform)      # two routes
        assert (dense - exact).norm() <= (transform - exact).norm()


@pytest.mark.gpu
@pytest.mark.parametrize("Lz,scale", [(1e23, 1e25), (1e12, 1.0), (1e-15, 1e-10)])
def test_dense_kernel_extreme_heights(api, Mr_5_25, Lz, scale):
    """Output factors 1 / dz and 1 / dz^2 that, with the operators' scale, leave float's range while the outputs do not."""
    import torch
    Nz, Ny, Nx = 513, 8, 2048
    z = np.arange(Nz) / (Nz - 1)
    f = (np.sin(np.outer(z, np.random.default_rng(1).uniform(3, 40, Ny * Nx)) + 1) * scale).astype(np.float32)
    ft = torch.from_numpy(f).cuda().view(1, Nz, Ny, Nx)
    plan = api.Plan(5, 25, Nz)
    out = [torch.empty_like(ft) for _ in range(2)]
    api.fc_deriv_z(plan, ft, *out, Lz=Lz)
    for order in (1, 2):
        err = np.linalg.norm(out[order - 1].view(Nz, -1)[:, :256].cpu().numpy() - _oracle(f[:, :256], Mr_5_25, order, Lz), axis=0)
        assert (err <= _bound(f[:, :256], Mr_5_25, order, Lz)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["peaks", "tiny"])
def test_dense_lines_do_not_depend_on_their_neighbours(api, kind):
    """The bits of a line are the same in any order of the lines, and in the slabs of a host call as in one call."""
    import torch
    Nz, Ny, Nx = 513, 10, 2050
    f = _field_with_peaks(Nz, Ny * Nx, 3)
    if kind == "tiny":
        f[:, ::97] *= np.float32(1e-36)
    ft = torch.from_numpy(f).cuda().view(1, Nz, Ny, Nx)
    plan = api.Plan(5, 25, Nz)
    d = [torch.empty_like(ft) for _ in range(2)]
    api.fc_deriv_z(plan, ft, *d)
    h = [torch.empty(ft.shape) for _ in range(2)]
    api.fc_deriv_z_host(plan, ft.cpu(), *h, slab_bytes=2 * Nz * Nx * 4)
    order = torch.randperm(Ny * Nx, generator=torch.Generator().manual_seed(1)).cuda()
    mixed = ft.view(Nz, -1)[:, order].contiguous().view(ft.shape)
    m = [torch.empty_like(ft) for _ in range(2)]
    api.fc_deriv_z(plan, mixed, *m)
    for a, b, c in zip(d, h, m):
        bits = a.view(torch.int32).view(Nz, -1)
        assert torch.equal(bits.cpu(), b.view(torch.int32).view(Nz, -1))
        assert torch.equal(bits[:, order], c.view(torch.int32).view(Nz, -1))


# ---------------------------------------------------------------------------
# float64: exact integer products (dense64.hpp)
# ---------------------------------------------------------------------------
def _lines64(Nz, n, seed):
    """Smooth and rough lines, wall layers, wide ranges of magnitude inside a line and between lines."""
    r = np.random.default_rng(seed)
    z = np.linspace(0, 1, Nz)[:, None]
    f = np.sin(z * r.uniform(1, 30, n) + 1) + r.uniform(-1, 1, n) * z ** 3
    f[:, 1::4] += 1e-3 * r.standard_normal((Nz, len(range(1, n, 4))))
    f[:, 2::4] = np.exp(-z * r.uniform(5, 60, len(range(2, n, 4)))) * 10.0 ** r.uniform(-200, 200, len(range(2, n, 4)))
    f[:, 3::4] *= np.where(np.arange(Nz) == Nz // 2, 1e6, 1.0)[:, None]
    return f


def _bound64(f, Mr, order, Lz=1.0):
    """Per line and value.  Line: whole units of at most 2^-52 of its largest value m, each off by half a unit, through an
    operator whose rows have 2-norm k_max^order (order 2: 0.45 of it) -> 2^-52 m k_max^order.  Operator: kernel values
    carry 2^-53 of themselves and whole units of 2^-54 of the largest, times at most m each -> 2^-52 sqrt(N') m k_max^order.
    Products left out and the outputs' units are below that; the same again for the rounding of the outputs and the sums
    of the two orders' scale factors."""
    m = np.abs(fc.extend(f, Mr)).max(axis=0)
    kmax = np.pi * (f.shape[0] - 1) / Lz
    return 4 * 2.0 ** -52 * np.sqrt(f.shape[0] + Mr.shape[0]) * m * kmax ** order


def _derivative_ld(f, Mr, order, Lz=1.0):
    """Continuation and derivative of f [Nz][lines] in extended precision."""
    ld = np.longdouble
    Nz, C, d = f.shape[0], Mr.shape[0], Mr.shape[1]
    Np = Nz + C
    x, M = f.astype(ld), Mr.astype(ld)
    cont = sum(M[:, i:i + 1] * x[Nz - d + i] + M[::-1, d - 1 - i:d - i] * x[i] for i in range(d))
    xe = np.vstack([x, cont])
    pi = ld("3.14159265358979323846264338327950288")
    k = np.arange(1, (Np + 1) // 2)
    ang = 2 * pi * ((np.arange(Np)[:, None] * k) % Np).astype(ld) / Np
    w = 2 * pi * k.astype(ld) / Np
    c = -2 * (w * np.sin(ang)).sum(1) if order == 1 else -2 * (w * w * np.cos(ang)).sum(1)
    if order == 2 and Np % 2 == 0:
        c = c - pi * pi * np.where(np.arange(Np) % 2, -1, 1)
    c = c / Np
    y = np.stack([(c[(n - np.arange(Np)) % Np][:, None] * xe).sum(0) for n in range(Nz)])
    return y / (ld(Lz) / (Nz - 1)) ** order


@pytest.mark.parametrize("Nz", [11, 20, 33, 39, 102, 103, 128, 231, 358, 513, 549])
def test_dense64_arithmetic_on_the_cpu(Nz, Mr_5_25):
    """The kernel's tables, index maps and number formats against the oracle, the digit sums below 2^24."""
    lib = _lib()
    f = np.ascontiguousarray(_lines64(Nz, 16, Nz))
    f[:, 15] = 0
    Mr = np.ascontiguousarray(Mr_5_25, dtype=np.float64)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    for order in (1, 2):
        y = np.full((Nz, 16), np.nan)
        assert lib.fchc_dense64_tile(Nz, 5, 25, ptr(Mr), order, ptr(f), ptr(y)) == 0
        err = np.abs(y - _derivative_ld(f, Mr, order, Nz - 1.0)).max(axis=0)
        bound = _bound64(f, Mr, order, Nz - 1.0)
        assert (err <= bound).all(), (order, (err / bound).max())
        assert not y[:, 15].any()


@pytest.mark.parametrize("d,C,Nz", [(3, 15, 40), (7, 33, 103), (10, 64, 201), (10, 64, 448), (4, 64, 512)])
def test_dense64_other_continuations_on_the_cpu(d, C, Nz):
    """test_dense64_arithmetic_on_the_cpu with other d and C, N' even and odd up to the largest.  The reference continues
    the lines in rational numbers: the weights of d = 10, C = 64 reach 1e10 and cancel."""
    from fractions import Fraction
    lib = _lib()
    from paper_2002_01392_gb300 import api as a
    f = np.ascontiguousarray(_lines64(Nz, 16, Nz))
    Mr = np.ascontiguousarray(a.Plan(d, C, Nz).matrix())
    M, F = [[Fraction(v) for v in row] for row in Mr.tolist()], [[Fraction(v) for v in row] for row in f.tolist()]

    def extended(v):   # to 64 bits
        hi = float(v)
        return np.longdouble(hi) + np.longdouble(float(v - Fraction(hi)))

    cont = np.array([[extended(sum(M[j][i] * F[Nz - d + i][n] + M[C - 1 - j][d - 1 - i] * F[i][n] for i in range(d)))
                      for n in range(16)] for j in range(C)])
    # the derivative of the line that is continued already: N' points, none added
    xe = np.vstack([f.astype(np.longdouble), cont])
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    for order in (1, 2):
        y = np.full((Nz, 16), np.nan)
        assert lib.fchc_dense64_tile(Nz, d, C, ptr(Mr), order, ptr(f), ptr(y)) == 0
        ref = _derivative_ld(xe, np.zeros((0, d)), order, Nz + C - 1.0)[:Nz]
        err = np.abs(y - ref).max(axis=0)
        assert (err <= _bound64(f, Mr, order, Nz - 1.0)).all()


def test_dense64_digit_sums_are_exact():
    """No sum of digit products of any operator that the float64 kernel takes can leave 2^24, where float32 still holds
    every whole number."""
    lib = _lib()
    lib.fchc_dense64_largest_sum.restype = ctypes.c_longlong
    most = [lib.fchc_dense64_largest_sum(Np - C, Np, order) for Np in range(6, 577) for C in (2, 3) for order in (1, 2)]
    assert sum(m > 0 for m in most) > 1800 and max(most) <= 2 ** 24


@pytest.mark.gpu
def test_given_up_waits_are_reported(api):
    """A kernel that gave up a wait (set on the host here) is reported once, by whatever call of the plan comes next, by the
    call itself where it is synchronous, or by fc_destroy; another plan is not concerned."""
    import torch
    Nz, Ny, Nx = 257, 8, 2560
    plan, other = api.Plan(5, 25, Nz), api.Plan(5, 25, Nz)
    f = torch.randn((1, Nz, Ny, Nx), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))

    def call(p, name, x):
        o = [torch.empty_like(x) for _ in range(2)]
        st = getattr(api._lib, name)(p.handle, api.FC_F32 if x.dtype == torch.float32 else api.FC_F64, 1, x.shape[3], x.shape[2],
                                     ctypes.c_double(1.0), x.data_ptr(), o[0].data_ptr(), o[1].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return st, o

    small, host = f[:, :, :1, :64].contiguous(), f.cpu()
    timeout = api.STATUS["FC_ERR_TIMEOUT"]
    good = call(plan, "fc_deriv_z", f)[1]
    for first in ("fc_deriv_z", "fc_deriv_z_noalloc"):
        for name, x in (("fc_deriv_z", small), ("fc_deriv_z", f.double()), ("fc_deriv_z_noalloc", f), ("fc_deriv_z_host", host)):
            api.inject_failure("dense_z_kernel", "FC_ERR_TIMEOUT")
            assert call(plan, first, f)[0] == 0
            assert call(other, name, x)[0] == 0
            assert call(plan, name, x)[0] == timeout and b"gave up" in api._lib.fc_last_error()
            assert call(plan, name, x)[0] == 0
    api.inject_failure("dense_z_kernel", "FC_ERR_TIMEOUT")
    assert call(plan, "fc_deriv_z_host", host)[0] == timeout
    st, o = call(plan, "fc_deriv_z_host", host)
    assert st == 0 and all(torch.equal(a, b.cpu()) for a, b in zip(o, good))
    api.inject_failure("dense_z_kernel", "FC_ERR_TIMEOUT")
    assert call(plan, "fc_deriv_z", f)[0] == 0
    assert api._lib.fc_destroy(plan.handle) == timeout
    plan.handle = None
    assert api._lib.fc_destroy(other.handle) == 0
    other.handle = None


@pytest.mark.gpu
def test_a_plans_first_call_prepares_all_others(api):
    """After one small call on a plan, large ones, of the other precision too, can be captured (what they add to the plan
    is no part of the graph), and fc_deriv_z_noalloc, whose tables are one precision's, only launches after a small call of the same."""
    import torch
    Nz, Ny, Nx = 513, 8, 2560
    plan = api.Plan(5, 25, Nz)
    f = torch.randn((1, Nz, Ny, Nx), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    ref = api.Plan(5, 25, Nz)
    for name in ("fc_deriv_z", "fc_deriv_z_noalloc"):
        for dt, code in ((torch.float32, api.FC_F32), (torch.float64, api.FC_F64)):
            x = f.to(dt)
            want = [torch.empty_like(x) for _ in range(2)]
            api.fc_deriv_z(ref, x, *want)
            small = x[:, :, :1, :64].contiguous()
            so, out = [torch.empty_like(small) for _ in range(2)], [torch.zeros_like(x) for _ in range(2)]

            def call(a, o):
                st = getattr(api._lib, name)(plan.handle, code, 1, a.shape[3], a.shape[2], ctypes.c_double(1.0), a.data_ptr(),
                                             o[0].data_ptr(), o[1].data_ptr(), torch.cuda.current_stream().cuda_stream)
                assert st == 0, api._lib.fc_last_error().decode()

            if name == "fc_deriv_z_noalloc" or dt == torch.float32:
                call(small, so)
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                call(x, out)
            call(x, out)       # not captured: whatever the capture would have copied is not there
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(out, want)), (name, dt)
            out[0].zero_()
            out[1].zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(out, want)), (name, dt)


@pytest.mark.gpu
@pytest.mark.parametrize("Nz,Ny,Nx,B,Lz", [(11, 5, 3, 1, 1.0), (33, 7, 37, 3, 2.0), (65, 64, 66, 1, 1.0), (102, 33, 31, 2, 1.0),
                                            (231, 48, 51, 1, 0.5), (358, 16, 17, 2, 1.0), (487, 48, 50, 1, 1.0), (513, 61, 41, 1, 1e-6),
                                            (549, 50, 49, 1, 1e5)])
def test_dense64_kernel(api, Mr_5_25, Nz, Ny, Nx, B, Lz):
    """Parts 4 and 2, tiles that end early or span fields, one output, wide magnitudes; NaN and Inf stay in their line;
    the entry points that route the same call agree bitwise."""
    import torch
    n = B * Ny * Nx
    f = np.ascontiguousarray(np.tile(_lines64(Nz, 64, Nz), (1, n // 64 + 1))[:, :n])
    bad = [n // 2] if n < 40 else [17, n // 2]
    f[Nz // 3, bad[0]] = np.nan
    f[0, bad[-1]] = np.inf if len(bad) > 1 else np.nan
    f[:, 3] = 0
    ft = torch.from_numpy(np.ascontiguousarray(f.reshape(Nz, B, Ny, Nx).transpose(1, 0, 2, 3))).cuda()
    plan = api.Plan(5, 25, Nz)
    d = [torch.full_like(ft, 7.0) for _ in range(2)]
    api.fc_deriv_z(plan, ft, *d, Lz=Lz)
    one = [torch.full_like(ft, 7.0) for _ in range(2)]
    api.fc_deriv_z(plan, ft, one[0], None, Lz=Lz)
    api.fc_deriv_z(plan, ft, None, one[1], Lz=Lz)
    noa = [torch.full_like(ft, 7.0) for _ in range(2)]
    assert api._lib.fc_deriv_z_noalloc(plan.handle, api.FC_F64, B, Nx, Ny, ctypes.c_double(Lz), ft.data_ptr(),
                                       noa[0].data_ptr(), noa[1].data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    h = [torch.empty(ft.shape, dtype=torch.float64) for _ in range(2)]
    api.fc_deriv_z_host(plan, ft.cpu(), *h, Lz=Lz, slab_bytes=2 * Nz * Nx * 8)
    torch.cuda.synchronize()
    good = np.setdiff1d(np.arange(n), bad)
    pick = np.unique(np.r_[good[:40], good[-20:]])
    for o in range(2):
        y = d[o].cpu().numpy().transpose(1, 0, 2, 3).reshape(Nz, n)
        assert np.isfinite(y[:, good]).all() and np.isnan(y[:, bad]).all() and not y[:, 3].any()
        err = np.abs(y[:, pick] - _derivative_ld(f[:, pick], Mr_5_25, o + 1, Lz)).max(axis=0)
        bound = _bound64(f[:, pick], Mr_5_25, o + 1, Lz)
        assert (err <= bound).all(), (o, np.nanmax(err / np.maximum(bound, 1e-300)))
        for other in (one[o], noa[o].cpu(), h[o]):
            z = other.cpu().numpy().transpose(1, 0, 2, 3).reshape(Nz, n)
            assert np.array_equal(z, y, equal_nan=True)
