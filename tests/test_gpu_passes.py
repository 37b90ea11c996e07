"""The passes over a whole field (energy, observables, render) at the sizes
where their work splits have edges: lattices smaller than a tile or a chunk of
planes, ragged sides, rows and planes one past a block, both z tiles."""
import ctypes

import numpy as np
import pytest

import bench
import oracle
import paper_2604_25876_gb300 as sk
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# smallest; one site past a 16- and a 32-wide z tile; odd rows; thin and long
SIZES = [(5, 5, 5), (6, 5, 21), (9, 20, 37), (7, 21, 20), (70, 13, 6), (12, 40, 53), (8, 6, 300)]


def field(n, h, seed=0, K=2):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(-0.3, 0.3, size=(K, 3))
    q = rng.normal(size=(K, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    return oracle.seed_product(n, h, pos, q, 0.8, False)


def on_gpu(phi, h, prec, **model):
    lat = sk.Lattice(phi.shape[:3], h, 1.0, prec, **model)
    st = sk.State(lat, DEV)
    sk.load_field(lat, st, phi)
    return lat, st, st.field().double().cpu().numpy()


def determinant_scale(phi, h):
    """Sum over the interior of the product of the determinant's row sizes /
    2 pi^2: |phi| and, for each derivative, its norm and |phi| / h (a stencil's
    rounding goes with the values it subtracts, not with their difference)."""
    prod = np.linalg.norm(phi, axis=-1)[2:-2, 2:-2, 2:-2]
    for ax in range(3):
        s = [phi.take(np.arange(2 + o, phi.shape[ax] - 2 + o), axis=ax) for o in (-2, -1, 1, 2)]
        d = (8 * (s[2] - s[1]) - (s[3] - s[0])) / (12 * h)
        keep = tuple(slice(None) if a == ax else slice(2, -2) for a in range(3))
        prod = prod * (np.linalg.norm(d, axis=-1)[keep] + 1.0 / h)
    return prod.sum() / (2 * np.pi ** 2)


# FP64: sums of at most 2e4 terms of one sign or of like size, each within a
# few eps64 of the oracle's.  FP32: a density's rounding is about 20 eps32 of
# its own size (stencil, products, minors), 1.2e-6, whatever the sums' signs.
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("prec,tol", [(64, 1e-12), (32, 2e-6)])
@pytest.mark.parametrize("model", [{}, {"m_y": 0.5, "m_z": 0.3, "m_w": 1.0, "c6": 0.7}])
def test_energy_matches_oracle_at_the_edges_of_the_work_split(n, prec, tol, model):
    h = 0.25
    lat, st, phi = on_gpu(field(n, h), h, prec, **model)
    om = oracle.Model(1.0, *model.values()) if model else 1.0
    eo, eg = oracle.energy(phi, h, om), sk.energy(lat, st)
    for k in ("E", "E2", "E4", "E0"):
        assert eg[k] == pytest.approx(eo[k], rel=tol, abs=tol * eo["E"]), k
    # (where the lattice is one site wide B is nothing but rounding)
    assert abs(eg["B"] - eo["B"]) <= tol * h ** 3 * determinant_scale(phi, h)
    assert eg["virial"] == pytest.approx(eo["virial"], abs=5 * tol * eo["E"])
    assert sk.energy(lat, st) == eg  # the same order every time


# potentials without the sextic term take the extended pass, whose sextic sum may
# overflow in FP32 on a field that is far from normalised: it counts for nothing
@pytest.mark.parametrize("model", [{"m_w": 1.0}, {"m_y": 0.3, "m_z": 0.2}])
def test_energy_without_the_sextic_term_does_not_overflow_with_it(model):
    n, h = (12, 13, 14), 0.25
    lat, st, phi = on_gpu(1e6 * field(n, h), h, 32, **model)
    om = oracle.Model(1.0, *(model.get(k, 0.0) for k in ("m_y", "m_z", "m_w", "c6")))
    eo, eg = oracle.energy(phi, h, om), sk.energy(lat, st)
    assert np.isfinite(list(eg.values())).all()
    # (E4 is a difference of terms of its size; E0 in FP32 takes 1 - phi^0 from the
    # pions of a unit field, so it is not the oracle's here)
    assert eg["E2"] == pytest.approx(eo["E2"], rel=2e-5)
    assert eg["E"] == pytest.approx(eg["E2"] + eg["E4"] + eg["E0"], rel=1e-12)


# (a lattice one site wide along an axis has no charge, so no observables)
@pytest.mark.parametrize("n", [(6, 7, 21), (9, 20, 37), (7, 21, 20), (70, 13, 8), (12, 40, 53),
                               (8, 9, 300)])
@pytest.mark.parametrize("prec", [64, 32])
def test_observables_match_oracle_at_the_edges_of_the_work_split(n, prec):
    h = 0.25
    lat, st, phi = on_gpu(field(n, h, 1), h, prec)
    o, g = oracle.observables(phi, h, 1.0), sk.observables(lat, st)
    # moments about X: scaled by the box and by |B|, which small boxes cut
    box = h * max(n)
    tol = (1e-10 if prec == 64 else 2e-6) * max(1.0, 1.0 / abs(o["B"]))
    for k in ("B", "E"):
        assert g[k] == pytest.approx(o[k], rel=tol), k
    assert np.allclose(g["X"], o["X"], atol=tol * box, rtol=0)
    for k in ("Q", "U", "V", "W"):
        a, b = np.array(g[k]), np.array(o[k])
        assert np.max(np.abs(a - b)) <= tol * max(1.0, np.max(np.abs(b))), k
    assert g["D"] == pytest.approx(o["D"], abs=tol * o["E"] * max(1.0, np.max(np.abs(o["V"]))))


# planes of so few sites that several runs along x share a block: one, some and
# many to a block, the last block's only partly there, one plane a run
# (a field cut so short that its mean square radius is negative has no R)
@pytest.mark.parametrize("n", [(6, 6, 6), (9, 6, 7), (61, 8, 9), (300, 6, 6), (300, 6, 7), (45, 12, 20), (30, 16, 15), (1300, 7, 8), (700, 20, 9),
                               (1217, 6, 7)])
@pytest.mark.parametrize("prec", [64, 32])
def test_observables_of_thin_lattices_match_oracle(n, prec):
    lat, st, phi = on_gpu(field(n, 0.25, 1), 0.25, prec)
    if np.isnan(oracle.observables(phi, 0.25, 1.0)["R"]):
        with pytest.raises(sk.SkyrmeError, match="non-finite"):
            sk.observables(lat, st)
        return
    test_observables_match_oracle_at_the_edges_of_the_work_split(n, prec)


def rotation(seed):
    q = np.random.default_rng(seed).normal(size=4)
    a, b, c, d = q / np.linalg.norm(q)
    return np.array([[a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c)],
                     [2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b)],
                     [2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d]])


@pytest.mark.parametrize("n", [(5, 6, 7), (33, 32, 35), (20, 90, 44), (66, 65, 64)])
@pytest.mark.parametrize("view", [None, 1, 2])
@pytest.mark.parametrize("levelset,scale,step", [(0.2, 4.0, 0.005), (0.6, 1.5, 0.011),
                                                 (1e-3, 3.0, 0.02), (0.0, 1.0, 0.03),
                                                 (0.3, -2.0, 0.02), (1.5, 4.0, 0.02)])
def test_whole_render_equals_the_plain_march_bit_for_bit(n, view, levelset, scale, step):
    """Samples passed over (by bricks, cells or the FP32 bound) change nothing:
    the whole render, the rays on its volume and the oracle's plain march of
    that volume give the same bits."""
    h = 0.25
    lat, st, _ = on_gpu(field(n, h, 4), h, 64)
    p = dict(width=50, height=37, view=None if view is None else rotation(view),
             levelset=levelset, transfer_scale=scale, step=step)
    img = sk.render(lat, st, sk.render_params(**p))
    vol = sk.render_volume(lat, st)
    assert torch.equal(img, sk.render_rays(vol, sk.render_params(**p)))
    ref = oracle.render_volume(vol.cpu().numpy(), **p).astype(np.float32)
    assert np.array_equal(img.cpu().numpy(), ref)


# rays of a few samples and of none, which the plain march takes behind the same
# tests of the box and the bricks: coarse steps, thin boxes face on and edge on,
# pictures of few and many pixels on either side of the choice
@pytest.mark.parametrize("n,view", [((33, 32, 35), None), ((33, 32, 35), 2), ((6, 90, 80), 1), ((6, 90, 80), None),
                                    ((80, 90, 6), None), ((5, 5, 5), 1)])
@pytest.mark.parametrize("levelset,scale,step", [(0.2, 4.0, 1.0), (0.2, 4.0, 0.2), (0.2, 4.0, 0.07), (1e-4, 4.0, 0.05),
                                                 (0.9, 30.0, 0.12), (0.0, 1.0, 0.5), (0.05, 4.0, 0.03)])
@pytest.mark.parametrize("width,height", [(13, 9), (400, 300)])
def test_rays_of_few_samples_equal_the_plain_march_bit_for_bit(n, view, levelset, scale, step, width, height):
    h = 0.25
    lat, st, _ = on_gpu(field(n, h, 4), h, 64)
    p = dict(width=width, height=height, view=None if view is None else rotation(view),
             levelset=levelset, transfer_scale=scale, step=step)
    for bright in (1.0, -2.0):
        p["brightness"] = bright
        img = sk.render(lat, st, sk.render_params(**p))
        vol = sk.render_volume(lat, st)
        assert torch.equal(img, sk.render_rays(vol, sk.render_params(**p)))
        ref = oracle.render_volume(vol.cpu().numpy(), **p).astype(np.float32)
        assert np.array_equal(img.cpu().numpy().view(np.int32), ref.view(np.int32))


def test_rays_pass_over_no_sample_that_is_not_finite():
    """Infinite and NaN densities count as the plain march counts them."""
    rng = np.random.default_rng(2)
    vol = rng.uniform(0.0, 0.15, size=(24, 22, 26, 4))
    vol[7, 8, 9, 0], vol[15, 11, 12, 0], vol[12, 5, 20, 0], vol[18, 18, 3, 0] = np.nan, np.inf, -np.inf, 0.9
    p = dict(width=61, height=47, levelset=0.2, step=0.01)
    img = sk.render_rays(torch.from_numpy(vol).to(DEV), sk.render_params(**p)).cpu().numpy()
    ref = oracle.render_volume(vol, **p).astype(np.float32)
    assert np.array_equal(img, ref, equal_nan=True)


def test_volume_quotients_are_correctly_rounded_over_the_range():
    """pion / |pion| of tiny, huge-ratio and denormal pions: IEEE quotients."""
    rng = np.random.default_rng(8)
    n = (12, 13, 14)
    phi = np.zeros(n + (4,))
    phi[..., 0] = 1.0
    mag = 10.0 ** rng.uniform(-300, 0, size=n + (3,))
    phi[..., 1:] = mag * rng.choice([-1.0, 1.0, 0.0], size=n + (3,))
    lat, st, got_phi = on_gpu(phi, 0.25, 64)
    vol = sk.render_volume(lat, st).cpu().numpy()
    ref = oracle.render_volume_from_field(got_phi, 0.25)
    assert np.array_equal(vol[..., 1:], ref[..., 1:])
    # an FP32 field with denormals (the widening's rare branch)
    lat, st, got_phi = on_gpu((10.0 ** rng.uniform(-44, 0, size=n + (4,))).astype(np.float32), 0.25, 32)
    vol = sk.render_volume(lat, st).cpu().numpy()
    ref = oracle.render_volume_from_field(got_phi, 0.25)
    assert np.array_equal(vol[..., 1:], ref[..., 1:])


# below and above the size from which the profile is tabulated; a constituent
# on a lattice site; radii past the table's last interval (rho = 57); a scale
# that is no power of two
@pytest.mark.parametrize("n,h,K,scale", [((9, 12, 33), 0.25, 3, 1.0), ((110, 100, 96), 0.3, 1, 0.5),
                                         ((101, 99, 103), 0.2, 2, 1.7)])
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("sym", [True, False])
def test_product_seed_matches_oracle(n, h, K, scale, prec, sym):
    rng = np.random.default_rng(K)
    pos = rng.uniform(-1.0, 1.0, size=(K, 3))
    pos[0] = [(n[a] // 2 - 0.5 * (n[a] - 1)) * h for a in range(3)]  # r = 0 at a site
    q = rng.normal(size=(K, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    lat = sk.Lattice(n, h, 1.0, prec)
    st = sk.State(lat, DEV)
    st.vel.fill_(3.0)
    sk.init_field(lat, sk.Seed.product(pos, q, scale, sym), st)
    ref = oracle.seed_product(n, h, pos, q, scale, sym)
    # 64 bits: a few eps per constituent, times the radius in the exponent
    # (symmetrised: over the norm of the sum, above 1e-3 here); 32: rounding
    got = st.phi[0].double().cpu().numpy()
    assert np.max(np.abs(got - ref)) <= (1e-12 if prec == 64 else 1.2e-7)
    assert torch.equal(st.phi[0], st.phi[1]) and not st.vel.any().item()
    assert sk.read_report(lat, st)["steps"] == 0


# sites taken 256 at a time across rows and planes: planes smaller than that,
# a last block of few sites, a single block
@pytest.mark.parametrize("n", [(5, 5, 5), (37, 6, 7), (300, 6, 6), (6, 5, 400)])
@pytest.mark.parametrize("prec", [64, 32])
def test_product_seed_of_thin_lattices_matches_oracle(n, prec):
    h, K = 0.25, 3
    rng = np.random.default_rng(1)
    pos, q = rng.uniform(-0.5, 0.5, size=(K, 3)), rng.normal(size=(K, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    lat = sk.Lattice(n, h, 1.0, prec)
    st = sk.State(lat, DEV)
    st.phi.fill_(3.0)
    st.vel.fill_(3.0)
    sk.init_field(lat, sk.Seed.product(pos, q, 1.0, True), st)
    ref = oracle.seed_product(n, h, pos, q, 1.0, True)
    assert np.max(np.abs(st.phi[0].double().cpu().numpy() - ref)) <= (1e-12 if prec == 64 else 1.2e-7)
    assert torch.equal(st.phi[0], st.phi[1]) and not st.vel.any().item()


# positions so far off that r^2 overflows (such a constituent is the vacuum),
# scales whose reciprocal overflows or is 0, and scales at the ends of the
# table's range; on both sides of the sizes from which the table and the
# double-float kernel are taken
@pytest.mark.parametrize("n,K", [((7, 9, 26), 2), ((64, 64, 64), 5)])
@pytest.mark.parametrize("far,scale", [(1e160, 1.0), (-3e300, 1.0), (0.0, 1e-309), (0.0, 1e-305),
                                       (0.0, 1e-90), (0.0, 1e90), (0.0, 1e300), (0.0, np.inf)])
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("sym", [True, False])
def test_product_seed_at_the_ends_of_the_number_range(n, K, far, scale, prec, sym):
    rng = np.random.default_rng(K)
    pos = rng.uniform(-1.0, 1.0, size=(K, 3))
    pos[0] = [(n[a] // 2 - 0.5 * (n[a] - 1)) * 0.25 for a in range(3)]  # r = 0 at a site
    pos[1] += [far, 0.0, -far]
    q = rng.normal(size=(K, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    lat = sk.Lattice(n, 0.25, 1.0, prec)
    st = sk.State(lat, DEV)
    sk.init_field(lat, sk.Seed.product(pos, q, scale, sym), st)
    ref = oracle.seed_product(n, 0.25, pos, q, scale, sym)
    assert np.isfinite(ref).all()
    got = st.phi[0].double().cpu().numpy()
    # as above: a few eps per constituent, or the FP32 rounding
    assert np.max(np.abs(got - ref)) <= (1e-12 if prec == 64 else 1.2e-7)


# the double-float kernel: rows of 24 sites, of one and a bit of a warp, a
# constituent on a site, radii on both sides of the table's ends (rho = 1/64
# and 32), many constituents, a coarse and a fine lattice
@pytest.mark.parametrize("n,h,K,scale", [((64, 64, 64), 0.15, 1, 1.0), ((47, 51, 24), 0.2, 8, 1.0),
                                         ((41, 60, 33), 0.02, 4, 1.0), ((60, 63, 95), 0.3, 2, 0.4),
                                         ((60, 40, 65), 1.0, 3, 2.5), ((28, 33, 35), 0.25, 64, 0.7)])
@pytest.mark.parametrize("sym", [True, False])
def test_large_fp32_product_seed_is_the_rounded_fp64_seed(n, h, K, scale, sym):
    rng = np.random.default_rng(K)
    pos = rng.uniform(-1.0, 1.0, size=(K, 3)) * min(2.0, 0.3 * h * min(n))
    pos[0] = [(n[a] // 2 - 0.5 * (n[a] - 1)) * h for a in range(3)]
    q = rng.normal(size=(K, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    phi = {}
    for prec in (32, 64):
        lat = sk.Lattice(n, h, 1.0, prec)
        st = sk.State(lat, DEV)
        st.vel.fill_(3.0)
        sk.init_field(lat, sk.Seed.product(pos, q, scale, sym), st)
        assert torch.equal(st.phi[0], st.phi[1]) and not st.vel.any().item()
        phi[prec] = st.phi[0].cpu()
    # both are within 1e-14 of the exact value (K = 64), so their roundings differ
    # only where it lies that close to the middle of two floats: 1e-14 / 6e-8 of
    # the components of size one (and as rarely of the others, whose errors
    # shrink with them), 0.2 of 1e6; then by one ulp
    ref = phi[64].float()
    off = phi[32] != ref
    assert int(off.sum()) <= 4
    assert torch.all((phi[32] - ref).abs()[off] <= 1.3e-7 * ref.abs()[off])


# where the force is NaN at some sites, delta is the largest of the others' (every
# lane, warp and CTA keeps its own), as the oracle's comparison passes over NaN
@pytest.mark.parametrize("n", [(12, 13, 14), (24, 26, 28)])
@pytest.mark.parametrize("prec,tol", [(64, 1e-10), (32, 1e-4)])
def test_delta_passes_over_sites_that_are_not_finite(n, prec, tol):
    h = 0.25
    phi = oracle.seed_rational_map(n, h, 2, 0.7)
    phi[n[0] // 2 - 1, n[1] // 2, n[2] // 2, 1] = np.nan  # among the strongest forces
    lat, st, phi = on_gpu(phi, h, prec)
    with pytest.raises(sk.SkyrmeError, match="non-finite"):
        sk.flow_step(lat, 1e-3, 1, sk.NEWTON, st)
    rep = sk.read_report(lat, st)
    _, f, _ = oracle.forces(phi, h, 1.0)
    ref = np.nanmax(np.linalg.norm(f, axis=-1))
    assert rep["delta"] == pytest.approx(ref, rel=tol) and np.isnan(rep["E"])


def captured_nodes(call):
    """How many kernels, copies and memsets ``call`` puts on its stream."""
    cu = ctypes.CDLL("libcuda.so.1")
    graph, s = torch.cuda.CUDAGraph(keep_graph=True), torch.cuda.Stream(DEV)
    with torch.cuda.graph(graph, stream=s):
        call()
    h, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert cu.cuGraphGetNodes(h, None, ctypes.byref(n)) == 0
    nodes, kind, count = (ctypes.c_void_p * n.value)(), ctypes.c_int(), [0, 0, 0]
    assert cu.cuGraphGetNodes(h, nodes, ctypes.byref(n)) == 0
    for node in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        count[kind.value] += 1
    return dict(zip(("kernels", "copies", "memsets"), count))


# The double-float kernel's margins, where products hand the scalar component the
# most error and where one constituent's vector is most of the site's; and only
# spacings at which the margins were measured take it (it clears its table).
@pytest.mark.parametrize("hs,radius,dominant,pairs", [(0.02, 0.3, False, True), (0.1, 0.0, False, True),
                                                      (0.1, 5.0, True, True), (0.0009, 0.01, False, False),
                                                      (0.001, 0.01, False, True)])
@pytest.mark.parametrize("sym", [True, False])
def test_fp32_product_seed_of_many_constituents(hs, radius, dominant, pairs, sym):
    n, scale, K = (40, 44, 45), 1.6, 64
    rng = np.random.default_rng(11)
    pos = rng.uniform(-1.0, 1.0, size=(K, 3)) * radius * scale
    if dominant:
        pos = np.sign(pos) * (0.6 * radius * scale + 0.4 * np.abs(pos))
        pos[K // 2] = [0.01, 0.0, -0.02]
    q = rng.normal(size=(K, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    phi = {}
    for prec in (32, 64):
        lat = sk.Lattice(n, hs * scale, 1.0, prec)
        st, seed = sk.State(lat, DEV), sk.Seed.product(pos, q, scale, sym)
        if prec == 32:
            assert captured_nodes(lambda: sk.init_field(lat, seed, st))["memsets"] == (1 if pairs else 0)
        sk.init_field(lat, seed, st)
        phi[prec] = st.phi[0].cpu()
    # as above: 1e-14 / 6e-8 of 3e5 values, one ulp each
    ref = phi[64].float()
    off = phi[32] != ref
    assert int(off.sum()) <= 4
    assert torch.all((phi[32] - ref).abs()[off] <= 1.3e-7 * ref.abs()[off])


# the FP64 step's columns (2 x 16 or 4 x 8), runs and shares: lattices of fewer
# units than warps, runs that cross columns, both column shapes, long runs
@pytest.mark.parametrize("n", SIZES + [(33, 48, 48), (200, 14, 18)])
@pytest.mark.parametrize("mode", [sk.ARRESTED, sk.NEWTON, sk.GRADIENT])
@pytest.mark.parametrize("model", [{}, {"m_y": 0.5, "m_z": 0.3, "m_w": 1.0, "c6": 0.02}])
def test_fp64_steps_match_oracle_at_the_edges_of_the_work_split(n, mode, model):
    h, dt, steps = 0.25, 0.004, 6
    lat, st, phi = on_gpu(field(n, h, 2), h, 64, **model)
    om = oracle.Model(1.0, *model.values()) if model else 1.0
    ost = oracle.new_state(phi)
    reps = oracle.flow(ost, h, om, dt, steps, mode=mode, reports=True)
    rep = sk.flow_step(lat, dt, steps, mode, st)
    # a few hundred roundings of the forces (up to 1e3 here) times dt, six steps
    assert np.max(np.abs(st.field().cpu().numpy() - ost.phi)) <= 1e-11
    if mode != sk.GRADIENT:
        scale = max(1.0, np.max(np.abs(ost.v)))
        assert np.max(np.abs(st.velocity().cpu().numpy() - ost.v)) <= 1e-11 * scale
    # (1 - phi^0 is rounded to eps of 1, not of itself: a converged field's
    # energy is a sum of such roundings)
    eps_sum = 1e-15 * h ** 3 * np.prod([v - 4 for v in n])
    for k in ("E", "E2", "E4", "E0"):
        assert rep[k] == pytest.approx(reps[-1][k], rel=1e-11, abs=1e-11 * reps[-1]["E"] + eps_sum), k
    assert rep["steps"] == steps and rep["status"] == 0


# several FP64 steps in a launch: fewer and more units than CTAs, both column
# shapes; time steps that arrest often, so that decisions are mispredicted
@pytest.mark.parametrize("n", [(7, 8, 21), (20, 22, 24), (24, 48, 48), (70, 66, 68)])
@pytest.mark.parametrize("mode,dt", [(sk.ARRESTED, 0.03), (sk.NEWTON, 0.004)])
def test_fp64_steps_of_one_call_equal_single_steps(n, mode, dt):
    h, steps = 0.25, 33
    lat, one, phi = on_gpu(field(n, h, 2), h, 64)
    _, many, _ = on_gpu(phi, h, 64)
    for _ in range(steps):
        a = sk.flow_step(lat, dt, 1, mode, one)
    b = sk.flow_step(lat, dt, steps, mode, many)
    assert a == b and b["steps"] == steps and b["status"] == 0
    assert torch.equal(one.phi, many.phi) and torch.equal(one.vel, many.vel)
    if mode == sk.ARRESTED and min(n) > 8:
        assert b["fixups"] > 0


# the corrections of several steps in one launch, by every entry point that
# runs them, for both instantiations of the step and both column shapes
@pytest.mark.parametrize("n", [(20, 22, 24), (24, 48, 48)])
@pytest.mark.parametrize("model,dt", [({}, 0.03), ({"m_y": 0.5, "m_z": 0.3, "m_w": 1.0, "c6": 0.02}, 0.02)])
@pytest.mark.parametrize("entry", ["call", "graph", "until"])
def test_fp64_corrections_in_a_launch_equal_single_steps(n, model, dt, entry):
    h, steps = 0.25, 60
    lat, one, phi = on_gpu(field(n, h, 2), h, 64, **model)
    _, many, _ = on_gpu(phi, h, 64, **model)
    for _ in range(steps):
        a = sk.flow_step(lat, dt, 1, sk.ARRESTED, one)
    if entry == "call":
        b = sk.flow_step(lat, dt, steps, sk.ARRESTED, many)
    elif entry == "graph":
        g = sk.FlowGraph(lat, many, dt, steps, sk.ARRESTED)
        g.launch()
        b = many.report()
        g.close()
    else:
        b = sk.flow_until(lat, dt, sk.ARRESTED, many, 0.0, steps, chunk=20)
    assert a == b and b["steps"] == steps and b["status"] == 0
    assert b["fixups"] > 1
    assert torch.equal(one.phi, many.phi) and torch.equal(one.vel, many.vel)


# as many steps to a launch as update 2^22 sites, and 128 at most
@pytest.mark.parametrize("n,steps,launches", [((8, 8, 8), 300, 3), ((24, 26, 28), 129, 2), ((24, 26, 28), 128, 1),
                                              ((48, 48, 48), 100, 3), ((170, 160, 180), 3, 3)])
@pytest.mark.parametrize("mode", [sk.ARRESTED, sk.NEWTON])
def test_fp64_steps_in_a_launch_are_capped(n, steps, launches, mode):
    lat = sk.Lattice(n, 0.25, 1.0, 64)
    st = sk.State(lat, DEV)
    sk.init_field(lat, sk.Seed.rational_map(1, 0.5), st)
    cl, cs = lat.c(), st.c()

    def call():
        rc = sk.load().skyrme_flow_step(ctypes.byref(cl), 0.004, steps, mode, ctypes.byref(cs), None,
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
    call()  # (a captured launch is not the first)
    torch.cuda.synchronize()
    assert captured_nodes(call) == {"kernels": launches, "copies": 0, "memsets": 0}
    wl = workloads.Workload("box", n, 0.25, 1.0, steps, 64, None, 0.004)
    assert bench.step_launches(wl, 64, steps) == launches


# Two flows on two streams at a time: FP64 launches that wait inside (for the
# arrest decision, for the next step), with one or two CTAs to an SM, some SMs
# idle, different lattices; and the modes whose launches do not wait.
@pytest.mark.parametrize("na,nb", [((48, 48, 48), (48, 48, 48)), ((20, 22, 24), (70, 66, 68)),
                                   ((70, 66, 68), (66, 70, 64))])
@pytest.mark.parametrize("prec,mode,dt", [(64, sk.ARRESTED, 0.03), (64, sk.NEWTON, 0.004), (64, sk.GRADIENT, 1e-5),
                                          (32, sk.NEWTON, 0.004), (32, sk.GRADIENT, 1e-5)])
def test_two_flows_on_two_streams_equal_the_flows_alone(na, nb, prec, mode, dt):
    h, steps, launches = 0.25, 40, 4
    pairs = [[on_gpu(field(n, h, 2 + k), h, prec)[:2] for k, n in enumerate((na, nb))] for _ in range(2)]
    for lat, st in pairs[0]:
        for _ in range(launches):
            sk.flow_step(lat, dt, steps, mode, st)
    graphs = [sk.FlowGraph(lat, st, dt, steps, mode) for lat, st in pairs[1]]
    torch.cuda.synchronize()
    for _ in range(launches):
        for g in graphs:
            with torch.cuda.stream(g.stream):  # each graph after its own last launch only
                g.launch()
    torch.cuda.synchronize()
    for (_, alone), (_, both) in zip(*pairs):
        rep = both.report()
        assert rep == alone.report() and rep["steps"] == steps * launches and rep["status"] == 0
        assert torch.equal(alone.phi, both.phi) and torch.equal(alone.vel, both.vel)
    for g in graphs:
        g.close()


def green_stream(sms):
    """A stream that owns about ``sms`` of the device's SMs, and how many it
    got (the driver's green contexts; its resource records are 144 bytes)."""
    cu = ctypes.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("the driver has no green contexts")
    torch.cuda.init()
    device, part, rest = (ctypes.create_string_buffer(1024) for _ in range(3))
    desc, ctx, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    count = ctypes.c_uint(1)
    for rc in (cu.cuDeviceGetDevResource(0, device, 1),
               cu.cuDevSmResourceSplitByCount(part, ctypes.byref(count), device, rest, 0, sms),
               cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
               cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, 0, 1),
               cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0)):
        assert rc == 0
    got = int.from_bytes(part.raw[96:100], "little")
    return cu, ctx, torch.cuda.ExternalStream(stream.value), got


# a stream that owns part of the SMs: launches that wait inside have to fit there
@pytest.mark.parametrize("mode,dt", [(sk.ARRESTED, 0.03), (sk.NEWTON, 0.004)])
@pytest.mark.parametrize("n", [(24, 48, 48), (70, 66, 68)])
def test_fp64_flow_on_a_stream_of_a_green_context(n, mode, dt):
    cu, ctx, s, sms = green_stream(32)
    assert 0 < sms < torch.cuda.get_device_properties(0).multi_processor_count
    h, steps = 0.25, 20
    lat, a, phi = on_gpu(field(n, h, 2), h, 64)
    _, b, _ = on_gpu(phi, h, 64)
    _, c, _ = on_gpu(phi, h, 64)
    torch.cuda.synchronize()
    ra, rb = sk.flow_step(lat, dt, steps, mode, a), sk.flow_step(lat, dt, steps, mode, b, stream=s)
    g = sk.FlowGraph(lat, c, dt, steps, mode, stream=s)
    with torch.cuda.stream(s):
        g.launch()
    s.synchronize()
    g.close()
    # the sums run over other shares of the lattice (rounding: 1e4 terms), the
    # sites' arithmetic is the same
    for r in (rb, c.report()):
        assert (r["steps"], r["arrests"], r["status"]) == (steps, ra["arrests"], 0)
        assert r["E"] == pytest.approx(ra["E"], rel=1e-12)
    assert torch.equal(a.phi, b.phi) and torch.equal(a.phi, c.phi)
    assert torch.equal(a.vel, b.vel) and torch.equal(a.vel, c.vel)
    assert cu.cuStreamDestroy_v2(ctypes.c_void_p(s.cuda_stream)) == 0 and cu.cuGreenCtxDestroy(ctx) == 0


@pytest.mark.parametrize("n", SIZES + [(6, 40, 52)])
@pytest.mark.parametrize("prec", [64, 32])
def test_load_field_gives_the_same_state_from_every_source(n, prec):
    """The direct read, the copy (host, other layout, other type, an offset
    that breaks the alignment, the state's own buffers) and the two outer
    layers, over the edges of the load kernel's blocks."""
    lat = sk.Lattice(n, 0.25, 1.0, prec)
    phi = field(n, 0.25, 3)
    ref = oracle.apply_vacuum_boundary(phi.copy())
    ref = torch.from_numpy(ref if prec == 64 else ref.astype(np.float32)).to(DEV)
    t = torch.from_numpy(phi).to(DEV, lat.dtype)
    odd = torch.empty(t.numel() + 1, dtype=lat.dtype, device=DEV)[1:].view(t.shape).copy_(t)
    sources = [t, phi, t.cpu(), t.transpose(0, 1).contiguous().transpose(0, 1), t.double(), odd,
               t.clone().requires_grad_(), -(-t)]
    for src in sources + ["own 0", "own 1"]:
        st = sk.State(lat, DEV)
        st.phi.fill_(0.5)
        st.vel.fill_(0.5)
        st.scratch.fill_(7)
        if isinstance(src, str):
            src, _ = st.phi[int(src[-1])], st.phi[int(src[-1])].copy_(t)
        with torch.no_grad():
            sk.load_field(lat, st, src)
        assert torch.equal(st.phi[0], ref) and torch.equal(st.phi[1], ref)
        assert not st.vel.any().item()
        rep = sk.read_report(lat, st)
        assert rep["steps"] == 0 and rep["cur"] == 0 and rep["status"] == 0
    with pytest.raises(RuntimeError):  # shapes that do not broadcast stay refused
        sk.load_field(lat, sk.State(lat, DEV), t[1:])


@pytest.mark.parametrize("n", [(5, 5, 5), (12, 40, 53)])
@pytest.mark.parametrize("prec", [64, 32])
def test_load_field_into_buffers_apart(n, prec):
    lat = sk.Lattice(n, 0.25, 1.0, prec)
    t = torch.from_numpy(field(n, 0.25, 3)).to(DEV, lat.dtype)
    ref = torch.from_numpy(oracle.apply_vacuum_boundary(t.double().cpu().numpy())).to(DEV, lat.dtype)
    st, wide = sk.State(lat, DEV), torch.zeros((4,) + t.shape, dtype=lat.dtype, device=DEV)
    st.phi = wide[::2]  # the source is the second of them
    wide[2].copy_(t)
    sk.load_field(lat, st, wide[2])
    assert torch.equal(wide[0], ref) and torch.equal(wide[2], ref) and not wide[1::2].any().item()
    st = sk.State(lat, DEV)  # tensors of their own
    st.phi, st.vel = [torch.empty_like(t) for _ in range(2)], [torch.empty_like(t) for _ in range(2)]
    sk.load_field(lat, st, t)
    assert torch.equal(st.phi[0], ref) and torch.equal(st.phi[1], ref)


def test_load_field_from_rejects_null_misaligned_and_overlapping_sources():
    import ctypes
    lat = sk.Lattice((6, 7, 8), 0.25, 1.0, 32)
    st = sk.State(lat, DEV)
    cl, cs = lat.c(), st.c()
    f = torch.zeros(6 * 7 * 8 * 4 + 4, device=DEV)
    call = lambda p: sk.load().skyrme_load_field_from(ctypes.byref(cl), ctypes.byref(cs),  # noqa: E731
                                                      ctypes.c_void_p(p), None)
    assert call(None) == 1 and call(f.data_ptr() + 4) == 1
    assert call(st.phi[0].data_ptr() + 16) == 1 and call(st.vel[1].data_ptr()) == 1
    assert call(f.data_ptr() + 16) == 0
    torch.cuda.synchronize()


# the load rewrites the control block while it reads its source, so a field in
# the state's scratch (where the control block is) goes through a copy
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("offset", [0, 8192])
def test_a_field_in_the_scratch_is_not_read_in_place(prec, offset):
    n = (6, 7, 8)
    lat = sk.Lattice(n, 0.25, 1.0, prec)
    st = sk.State(lat, DEV)
    t = torch.from_numpy(field(n, 0.25, 3)).to(DEV, lat.dtype)
    nbytes = t.numel() * t.element_size()
    src = st.scratch[offset:offset + nbytes].view(lat.dtype).view(t.shape)
    cl, cs = lat.c(), st.c()
    rc = sk.load().skyrme_load_field_from(ctypes.byref(cl), ctypes.byref(cs),
                                          ctypes.c_void_p(src.data_ptr()), None)
    assert rc == 1
    src.copy_(t)
    sk.load_field(lat, st, src)
    ref = torch.from_numpy(oracle.apply_vacuum_boundary(t.double().cpu().numpy())).to(DEV, lat.dtype)
    assert torch.equal(st.phi[0], ref) and torch.equal(st.phi[1], ref) and not st.vel.any().item()
    assert sk.read_report(lat, st)["steps"] == 0
