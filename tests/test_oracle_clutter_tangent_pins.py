"""Pins of the oracle's clutter measure where an edge of a triangle only touches the cylinder, at its middle
(where a piece between two crossings has its own middle), and where it passes through the axis.
"""
import numpy as np
import pytest


def area(tri, R=1.0):
    import oracle

    v = np.concatenate([np.asarray(tri, np.float32), np.zeros((1, 3), np.float32)])
    n = np.zeros_like(v)
    n[-1, 2] = 1
    return float(oracle.clutter_areas(v, n, np.array([[0, 1, 2]], np.int32), [3], R, 3)[0][0])


def test_an_edge_that_touches_from_outside_adds_nothing():
    assert area([(-1, -0.75, 0), (-1.5, -1, 0.25), (-1, 0.75, 0.25)]) == pytest.approx(0, abs=1e-15)
    assert area([(1, -0.5, 0), (1, 0.5, 0), (1.5, 0, 0.25)]) == pytest.approx(0, abs=1e-15)


def test_an_edge_that_touches_from_inside_cuts_nothing_off():
    # the half disk x >= 0, its far edge along x = 1
    tri = [(1, -4, 0), (1, 4, 0), (-1, 0, 0)]
    inside = area(tri)
    wider = area([(1.5, -5, 0), (1.5, 5, 0), (-1, 0, 0)])  # the same two other edges
    assert inside == pytest.approx(wider, rel=1e-14)


def test_an_edge_through_the_axis():
    """Half of a band: values by numerical integration of the chord (20,000 steps)."""
    assert area([(0.5, 1.5, -3), (-0.5, -1.5, 2), (-1, -1, 0.5)]) == pytest.approx(0.715667369, rel=1e-7)
