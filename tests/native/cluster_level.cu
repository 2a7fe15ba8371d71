// The choice of the cluster level with a stand-in for the device's answer: a cluster can be placed when a CTA
// needs at most `limit` bytes.
#include "mg_common.cuh"

extern "C" int pick_cluster_level(const int *n, int nlev, int robin, int tb, long long limit)
{
    std::vector<ctt::Geo> lev(nlev);
    for (int l = 0; l < nlev; ++l)
        for (int a = 0; a < 3; ++a) lev[l].n[a] = n[a] >> l;
    return ctt::cluster_level(lev.data(), nlev, robin, (size_t)tb, [&](size_t bytes) { return (long long)bytes <= limit; });
}
