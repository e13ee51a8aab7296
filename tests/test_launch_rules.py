"""The host-side rules that choose a launch's form (csrc/rc_rules.h), compiled
by themselves and called on the CPU."""
import numpy as np
import pytest

from launch_rules import compile_rules, launch_size, view


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    return compile_rules(tmp_path_factory.mktemp("rules"))


DIMS, ONES = (256, 256, 180), (1.0, 1.0, 1.0)
CENTRE = (127.5, 127.5, 89.5)


def orbit(n, size, dist=800.0):
    a = np.radians(12.0 + 360.0 * np.arange(n) / n)
    return [view(DIMS, ONES, (127.5 + dist * np.cos(x), 127.5 + dist * np.sin(x), 89.5 + 0.35 * dist), CENTRE, size) for x in a]


# a chunk gets an SM of its own before two share one
@pytest.mark.parametrize("chunks,ctas", [(1, 1), (3, 3), (64, 64), (151, 151), (152, 152), (153, 152), (456, 152),
                                         (1 << 27, 152)])
def test_a_small_image_spreads_over_the_sms(rules, chunks, ctas):
    assert rules.persistent_ctas(chunks, 152) == ctas


def orbit_size(rules, dims, size, views, step):
    """Size of a launch of `views` square views on the orbit that just holds the box."""
    ext = np.array(dims) - 1.0
    dist = 1.1 * np.linalg.norm(ext) / 2 / np.sin(np.radians(15.0))
    el, az = np.radians(20.0), np.radians(12.0 + 360.0 * np.arange(views) / views)
    return launch_size(rules, dims, ONES, step, [
        view(dims, ONES, ext / 2 + dist * np.array([np.cos(el) * np.cos(a), np.cos(el) * np.sin(a), np.sin(el)]), ext / 2,
             (size, size)) for a in az])


# a view that looks past the volume or stands far from it changes a launch's
# size by its own rays only, wherever it stands among the views
@pytest.mark.parametrize("other", [view(DIMS, ONES, (827.5, 127.5, 89.5), (327.5, 1027.5, 89.5), (1024, 1024)),
                                   view(DIMS, ONES, (9127.5, 127.5, 89.5), CENTRE, (1024, 1024))])
def test_every_view_counts(rules, other):
    views = orbit(7, (1024, 1024))
    base, steps, _ = launch_size(rules, DIMS, ONES, 0.5, views)
    assert 150e3 * 7 < base < 600e3 * 7
    for at in (0, 3, 7):
        hits, s, density = launch_size(rules, DIMS, ONES, 0.5, views[:at] + [other] + views[at:])
        assert abs(hits - base) < 5e3 and s == steps
        assert rules.lanes_per_ray(hits, s, 0) == 1 and rules.lanes_per_sum(hits, s, density, 0) == 1
    alone, s, _ = launch_size(rules, DIMS, ONES, 0.5, [other])
    assert alone < 5e3 and rules.lanes_per_ray(alone, s, 0) == 8


# many views are sized by a spread sample of them
def test_many_views_are_sampled(rules):
    one, steps, density = launch_size(rules, DIMS, ONES, 0.5, orbit(1, (64, 64)))
    for n in (32, 33, 1000, 65535):
        hits, s, d = launch_size(rules, DIMS, ONES, 0.5, orbit(n, (64, 64)))
        assert s == steps and 0.7 * density < d < 1.4 * density and 0.7 * n * one < hits < 1.4 * n * one


# (dims, image, views, step): lanes of the trilinear and the B-spline sums where
# the measured times leave one answer (another is slower by 15% or more): short
# chains and pixels dense on the voxels take fewer
@pytest.mark.parametrize("dims,size,views,step,lanes", [
    ((256, 256, 180), 128, 1, 0.5, (4, 4)), ((128, 128, 96), 128, 1, 10.0, (4, 4)),
    ((128, 128, 96), 512, 1, 20.0, (1, None)), ((128, 128, 96), 724, 1, 10.0, (1, 1)),
    ((64, 64, 32), 1024, 1, 0.5, (1, None)), ((40, 40, 40), 1024, 1, 0.5, (1, 1)),
    ((40, 40, 40), 1024, 1, 2.0, (1, 1)), ((256, 256, 180), 1024, 1, 0.5, (2, None)),
    ((256, 256, 180), 1024, 4, 0.5, (None, 2)), ((256, 256, 180), 1024, 8, 0.5, (None, 2)), ((51, 302, 86), 870, 4, 0.5, (2, None))])
def test_lanes_of_sums(rules, dims, size, views, step, lanes):
    z = orbit_size(rules, dims, size, views, step)
    for cubic in (0, 1):
        if lanes[cubic]:
            assert rules.lanes_per_sum(*z, cubic) == lanes[cubic], (cubic, z)


# the same for maxima
@pytest.mark.parametrize("dims,size,views,step,lanes", [
    ((256, 256, 180), 128, 1, 0.5, (4, 4)), ((256, 256, 180), 256, 1, 0.5, (4, 4)),
    ((512, 512, 256), 512, 2, 0.5, (4, 4)), ((128, 128, 96), 1024, 8, 0.5, (1, None)),
    ((64, 64, 32), 1448, 1, 0.5, (1, None)), ((256, 256, 180), 1024, 8, 0.5, (2, 2)),
    ((51, 302, 86), 1024, 4, 0.5, (None, 2))])
def test_lanes_of_maxima(rules, dims, size, views, step, lanes):
    z = orbit_size(rules, dims, size, views, step)
    for cubic in (0, 1):
        if lanes[cubic]:
            assert rules.lanes_per_max(*z, cubic) == lanes[cubic], (cubic, z)


# from inside the box every pixel has a ray, and its chain is short
@pytest.mark.parametrize("size,lanes", [(64, 8), (128, 4), (256, 1), (1024, 1)])
def test_lanes_inside_the_box(rules, size, lanes):
    eye, target = (102.4, 115.2, 90.0), (230.4, 128.0, 108.0)
    hits, steps, density = launch_size(rules, DIMS, ONES, 0.5, [view(DIMS, ONES, eye, target, (size, size), fovy=60.0)])
    assert hits == size * size
    outside = launch_size(rules, DIMS, ONES, 0.5, orbit(1, (size, size)))[1]
    assert 0.3 * outside < steps < 0.4 * outside
    assert rules.lanes_per_ray(hits, steps, 0) == lanes
    assert rules.lanes_per_sum(hits, steps, density, 0) == {64: 4, 128: 4, 256: 4, 1024: 1}[size]
