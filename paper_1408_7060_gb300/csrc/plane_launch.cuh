// Launches of the plane kernel, dispatched over the padded lengths, and its set-up; one
// translation unit per precision.
#pragma once
#include <algorithm>

#include "operator_impl.cuh"

template <int L, class F>
static void plane_with_z(int lz, F&& f) {
  with_zlen(lz, [&](auto z) {
    if constexpr (decltype(z)::value <= L) f(z);
    else throw AimError{AIM_ERR_ARG, "z transform longer than the padded length"};
  });
}
template <class F>
static void plane_with_l(int l, F&& f) {
  switch (l) {
    case 16: f(std::integral_constant<int, 16>{}); break;
    case 32: f(std::integral_constant<int, 32>{}); break;
    case 64: f(std::integral_constant<int, 64>{}); break;
    case 128: f(std::integral_constant<int, 128>{}); break;
    case 192: f(std::integral_constant<int, 192>{}); break;
    case 256: f(std::integral_constant<int, 256>{}); break;
    default: throw AimError{AIM_ERR_ARG, "plane kernel: padded length"};
  }
}

template <class C>
void plane_launch(aim_ctx* c, int nb, int mode, int m, const int* active, C* S, int slots, size_t slot_elems) {
  plane_with_l(c->L, [&](auto lt) {
    constexpr int L = decltype(lt)::value;
    plane_with_z<L>(c->LZ, [&](auto zt) {
      constexpr int LZ = decltype(zt)::value;
      if constexpr (plane_fits<L, LZ, C>()) {
        PlaneArgs<C> a{reinterpret_cast<C*>(c->d_A), S, sel_plane(c, (C*)nullptr), nb * 4, slot_elems, active,
                       sel_tw(c, (C*)nullptr), sel_twz(c, (C*)nullptr), c->NZ};
        a.G += (size_t)m * plane_spec_elems(plane_order<L, LZ, C>());
        constexpr size_t sm = PlaneCfg<L, LZ, C>::smem;
        auto go = [&](auto kern) {
          smem_opt_in(kern, sm);
          launch_pdl(c->stream, dim3(slots * nb * 4, L), dim3(32 * PlaneCfg<L, LZ, C>::NW), sm, kern, a);
        };
        switch (mode) {
          case PLANE_CONV: go(k_plane<L, LZ, C, PLANE_CONV>); break;
          case PLANE_FWD: go(k_plane<L, LZ, C, PLANE_FWD>); break;
          default: go(k_plane<L, LZ, C, PLANE_INV>);
        }
      } else {
        throw AimError{AIM_ERR_ARG, "plane kernel: the plane does not fit shared memory"};
      }
    });
  });
}

// the delay sum over z-spectra into S, then through the plane kernel's inverse into d_A
template <class C>
void plane_rhs(aim_ctx* c, int nb, const SlabList& sl, C* S) {
  plane_with_l(c->L, [&](auto lt) {
    constexpr int L = decltype(lt)::value;
    plane_with_z<L>(c->LZ, [&](auto zt) {
      constexpr int LZ = decltype(zt)::value;
      if constexpr (plane_fits<L, LZ, C>()) {
        const long long pairs = (long long)L * L * LZ / 2;
        k_spec_sum<C><<<dim3((unsigned)((pairs + 255) / 256), nb * 4), 256, 0, c->stream>>>(
            sl, sel_plane(c, (C*)nullptr), plane_order<L, LZ, C>(), S);
        AIM_CHECK_LAUNCH();
      }
    });
  });
  plane_launch<C>(c, nb, PLANE_INV, 0, nullptr, S, 1, 0);
}

// Whether a plane of this context's size fits shared memory, and the order of its spectra.
template <class C>
static bool plane_order_of(const aim_ctx* c, PlaneOrder* o) {
  if (c->L > 256) return false;
  bool fits = false;
  plane_with_l(c->L, [&](auto lt) {
    constexpr int L = decltype(lt)::value;
    plane_with_z<L>(c->LZ, [&](auto zt) {
      constexpr int LZ = decltype(zt)::value;
      if constexpr (plane_fits<L, LZ, C>()) {
        fits = true;
        *o = plane_order<L, LZ, C>();
      }
    });
  });
  return fits;
}
template <class C>
bool plane_holds(const aim_ctx* c) {
  PlaneOrder o{};
  return plane_order_of<C>(c, &o);
}

// The plane kernel's spectra of nm delays from the octants.
template <class C>
C* plane_tables(aim_ctx* c, int nm, const C* oct) {
  PlaneOrder o{};
  if (!plane_order_of<C>(c, &o)) throw AimError{AIM_ERR_ARG, "plane kernel: the plane does not fit shared memory"};
  const size_t per = plane_spec_elems(o);
  C* g = (C*)aim_alloc(c, (size_t)nm * per * sizeof(C));
  const size_t no = 2 * (size_t)(c->N + 1) * (c->N + 1) * (c->LZ / 2 + 1);
  for (int m = 0; m < nm; ++m) {
    k_plane_spec<C><<<(int)std::min<size_t>((per + 255) / 256, 152 * 16), 256, 0, c->stream>>>(
        o, oct + m * no, g + m * per);
    AIM_CHECK_LAUNCH();
  }
  return g;
}
